"""The two streams of a step: what a step leaves pending never reaches the next one late.  Each case enqueues its steps
behind other work, so that the host is far ahead of the device, and again with a synchronisation before every
step: the same bits."""

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _hidden(n, D, seed):
    g = np.random.default_rng(9300 + seed)
    return W.to_bf16_grid(g.standard_normal((n, D)).astype(np.float32))


def _layers(n, budget, kv_dtype, d=64, D=256):
    from paper_2410_01805_b200 import LocretLayer
    from parity_util import bf16_dev
    sh = W.LayerShape(d_model=D, n_q_heads=4, n_kv_heads=2, head_dim=d, d_retain=128, rope_theta=500000.0, kv_dtype=kv_dtype)
    return sh, [LocretLayer(sh, *(bf16_dev(a) for a in W.layer_weights(sh, i, seed=W.BASE_SEED + 23)), budget, 300, 16, reserve=200)
                for i in range(n)]


def _both_ways(run):
    """run(wait): enqueues the steps, calling wait() between them; returns tensors and states."""
    busy = torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16)
    got = []
    for synchronised in (True, False):
        torch.cuda.synchronize()
        if not synchronised:
            for _ in range(40):       # a few milliseconds for the host to run ahead
                torch.mm(busy, busy)
        outs, layers = run(torch.cuda.synchronize if synchronised else lambda: None)
        assert all(L.sync_status() == 0 for L in layers)
        got.append((outs, [L.export_state() for L in layers]))
        for L in layers:
            L.destroy()
    (a, sa), (b, sb) = got
    assert torch.equal(a, b)
    for x, y in zip(sa, sb):
        for key in x:
            assert np.array_equal(x[key], y[key]), key


@pytest.mark.parametrize("how", ["calls", "stack", "evicting"])
@pytest.mark.parametrize("n_last", [45, 300])
def test_four_bit_chunk_after_one_token_steps(how, n_last):
    """The chunk's expansion reads the codes, scales and ranks that the token steps before it wrote."""
    from paper_2410_01805_b200 import LayerStack, NO_EVICT
    from parity_util import bf16_dev

    def run(wait):
        sh, layers = _layers(2, 200, 1)
        width = sh.n_q_heads * sh.head_dim
        first, tokens, last = (bf16_dev(_hidden(n, sh.d_model, i)) for i, n in enumerate((200, 100, n_last)))
        out = torch.zeros((2, 300, width), dtype=torch.bfloat16, device="cuda")
        one = torch.zeros((2, width), dtype=torch.bfloat16, device="cuda")
        stack = LayerStack(layers)
        for L in layers:
            L.prefill_chunk(first, out[0, :200], 0)
        for t in range(100):
            wait()
            if how == "stack":
                stack.decode_step(tokens[t], one, out_stride=width)
            else:
                for i, L in enumerate(layers):
                    L.prefill_chunk(tokens[t:t + 1], one[i], 0 if how == "evicting" else NO_EVICT)
        wait()
        for i, L in enumerate(layers):
            L.prefill_chunk(last, out[i, :n_last], 0)
        return out, layers

    _both_ways(run)


def test_four_bit_chunk_after_a_step_on_one_stream():
    """A step that keeps every kernel on the layer's stream (timing mode 2) reads the expansion scratch there; the next
    step, of another layer, fills the scratch on the second stream."""
    from paper_2410_01805_b200 import NO_EVICT
    from parity_util import bf16_dev

    def run(wait):
        sh, layers = _layers(2, 400, 1)
        x = [bf16_dev(_hidden(300, sh.d_model, 70 + i)) for i in range(3)]
        out = torch.zeros((2, 300, sh.n_q_heads * sh.head_dim), dtype=torch.bfloat16, device="cuda")
        for L in layers:
            L.prefill_chunk(x[0], out[0], NO_EVICT)
        wait()
        layers[0].set_timing(2)
        layers[0].prefill_chunk(x[1], out[0], NO_EVICT)
        wait()
        layers[1].prefill_chunk(x[2][:40], out[1, :40], NO_EVICT)
        return out, layers

    _both_ways(run)


@pytest.mark.parametrize("kv_dtype", [0, 1])
@pytest.mark.parametrize("n_layers", [1, 2])
def test_chunks_that_evict_and_chunks_that_do_not(kv_dtype, n_layers):
    """A chunk's projection starts beside its layer's last retaining head if that step did not evict, and after its
    compaction if it did; one-token steps between them run on the layer's own stream."""
    from paper_2410_01805_b200 import NO_EVICT
    from parity_util import bf16_dev

    def run(wait):
        sh, layers = _layers(n_layers, 500, kv_dtype)
        sizes = [(300, 0), (150, NO_EVICT), (300, 0), (40, NO_EVICT), (1, 0), (300, 0), (300, 0), (1, NO_EVICT), (64, NO_EVICT),
                 (200, 0), (130, NO_EVICT), (20, 0)]   # (the third evicts the first 250 of 750 units)
        out = torch.zeros((n_layers, sum(n for n, _ in sizes), sh.n_q_heads * sh.head_dim), dtype=torch.bfloat16, device="cuda")
        x = bf16_dev(_hidden(out.shape[1], sh.d_model, 80))
        t = 0
        for n, flags in sizes:
            for i, L in enumerate(layers):
                wait()
                L.prefill_chunk(x[t:t + n], out[i, t:t + n], flags)
            t += n
        return out, layers

    _both_ways(run)
