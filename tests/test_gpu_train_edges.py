"""Training kernels at the edges of their tiles: labels (query tiles of gb heads x 256 / gb answers, pairs of
128 keys, work units that divide the query tiles), loss and gradients (column tiles, slabs of tokens, heads
padded to 8 or 32), AdamW (vectors of four and the remainder)."""

import numpy as np
import pytest
import torch

import workloads as W
from oracle import locret_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_a,n_q,h,hk,d", [(64, 256, 4, 1, 128), (65, 257, 16, 1, 64), (16, 255, 32, 1, 96),
                                            (130, 511, 12, 2, 128), (300, 33, 5, 5, 64), (1024, 700, 4, 1, 96)])
def test_labels_at_tile_edges(n_a, n_q, h, hk, d):
    from parity_util import bf16_dev
    from paper_2410_01805_b200 import cis_labels
    g = np.random.default_rng(n_a + n_q)
    q = W.to_bf16_grid((g.standard_normal((n_a, h, d)) - 0.3).astype(np.float32))
    k = W.to_bf16_grid(np.abs(g.standard_normal((n_q, hk, d))).astype(np.float32))  # mostly negative products
    ref = O.cis_labels(q, k, hk, 1.0)
    got = cis_labels(bf16_dev(q), bf16_dev(k)).cpu().numpy().astype(np.float64)
    # exact bf16 products, d <= 128 fp32 additions: d * 2^-24 relative to sum |q k|, which is below 4 d here
    assert np.abs(got - ref).max() <= d * 2.0 ** -24 * 4 * d


@pytest.mark.parametrize("n,d_in,d_R,hk", [(64, 64, 32, 1), (192, 192, 96, 9), (320, 64, 288, 8), (128, 320, 160, 32)])
def test_loss_and_gradients_at_tile_edges(n, d_in, d_R, hk):
    from test_gpu_train import test_loss_and_gradients_match_the_oracle
    test_loss_and_gradients_match_the_oracle(n, d_in, d_R, hk)


def test_the_training_call_has_its_own_status_word():
    """Calls may overlap: the word that a timed-out wait writes lies in the call's workspace, cleared by the call."""
    import ctypes
    import paper_2410_01805_b200 as P
    n, d_in, d_R, hk = 64, 64, 32, 2
    need = ctypes.c_int64()
    assert P.lib.locret_rh_loss_grad_workspace(n, d_R, hk, ctypes.byref(need)) == 0
    ws = torch.full((need.value,), 0xFF, dtype=torch.uint8, device="cuda")
    z, w1, w2 = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((n, d_in), (d_in, d_R), (d_R, hk)))
    lab, loss, g1, g2 = (torch.zeros(s, device="cuda") for s in ((hk, n), (1,), (d_in, d_R), (d_R, hk)))
    args = [t.data_ptr() for t in (z, lab, w1, w2)] + [n, d_in, d_R, hk, 0.1] + [t.data_ptr() for t in (loss, g1, g2, ws)]
    st = torch.cuda.current_stream().cuda_stream
    assert P.lib.locret_rh_loss_grad_ws(*args, need.value, st) == 0
    assert ws[-256:-252].tolist() == [0, 0, 0, 0] and ws[-252:].eq(0xFF).all()
    assert P.lib.locret_rh_loss_grad_ws(*args, need.value - 1, st) == -3


@pytest.mark.parametrize("n,offset", [(1, 0), (4, 0), (1027, 0), (1024, 1), (1030, 2)])
def test_adamw_vectors_and_remainder(n, offset):
    from paper_2410_01805_b200 import adamw_step
    g = torch.Generator().manual_seed(n)
    a = [torch.randn(n + offset, generator=g, dtype=torch.float64).float()[offset:] for _ in range(4)]
    a[3] = a[3].abs()
    dev = [torch.empty(n + offset, device="cuda")[offset:].copy_(t) for t in a]
    b16 = torch.zeros(n + offset, dtype=torch.bfloat16, device="cuda")[offset:]
    adamw_step(dev[0], dev[1], dev[2], dev[3], 3, 5e-4, param_bf16=b16)
    p, gr, m, v = (t.double() for t in a)
    m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
    ref = p * (1 - 5e-4 * 0.01) - 5e-4 * (m / (1 - 0.9 ** 3)) / ((v / (1 - 0.999 ** 3)).sqrt() + 1e-8)
    # a dozen fp32 roundings of values of order one, and the update's rounded constants (lr / bias terms: 1e-5 of 5e-4)
    assert (dev[0].cpu().double() - ref).abs().max() <= 16 * 2.0 ** -24 * max(1.0, float(ref.abs().max()))
    assert torch.equal(b16, dev[0].bfloat16())


def test_calls_of_several_threads():
    """Labels and training calls of eight host threads, each on a stream of its own: the results of the same calls alone."""
    import threading
    from parity_util import bf16_dev
    from paper_2410_01805_b200 import cis_labels, rh_loss_grad
    g = np.random.default_rng(31)
    work = []
    for i in range(8):
        n = 512 + 64 * i
        q, k = bf16_dev(g.standard_normal((40 + i, 4, 64))), bf16_dev(g.standard_normal((n, 2, 64)))
        z, w1, w2 = bf16_dev(g.standard_normal((n, 128))), bf16_dev(g.standard_normal((128, 64)) / 11), bf16_dev(g.standard_normal((64, 2)) / 8)
        labels = cis_labels(q, k)
        work.append(((q, k), (z, w1, w2), labels, rh_loss_grad(z, labels, w1, w2)))
    torch.cuda.synchronize()
    bad = []

    def run(i):
        (q, k), (z, w1, w2), labels, (loss, d_w1, d_w2) = work[i]
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(20):
                    assert torch.equal(cis_labels(q, k), labels)
                    a, b, c = rh_loss_grad(z, labels, w1, w2)
                    assert torch.equal(b, d_w1)
                    # loss and dW2 are summed with fp32 atomics: n additions in any order
                    assert abs(float(a - loss)) <= 1e-5 * abs(float(loss)) and float((c - d_w2).abs().max()) <= 1e-5 * float(d_w2.abs().max())
        except Exception as e:   # (seen by the thread that waits)
            bad.append((i, repr(e)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
