"""The per-thread cache of tensor maps: a GEMM whose one operand has been in the cache for long while the other takes a new
slot, at every position of the slot that is reused next."""

import threading

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tok", [64, 600])   # the projection of few tokens, and the wide GEMM
def test_an_old_map_beside_a_new_one(n_tok):
    import paper_2410_01805_b200 as P
    from parity_util import bf16_dev
    d_in, d_R, n_w = 64, 64, 600                # more than twice the cache's slots
    g = np.random.default_rng(5)
    z = bf16_dev(g.standard_normal((n_tok, d_in)))
    w1 = bf16_dev(g.standard_normal((n_w, d_R, d_in)) / 8)
    w2 = torch.from_numpy(W.to_bf16_grid((g.standard_normal((d_R, 1)) / 8).astype(np.float32))).cuda()
    got = torch.full((n_w, n_tok), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = []

    def run():   # (a thread of its own: the cache starts empty)
        torch.cuda.set_device(0)
        st = torch.cuda.current_stream().cuda_stream
        for i in range(n_w):
            rc.append(P.lib.locret_rh_scores_static(z.data_ptr(), n_tok, d_in, w1[i].data_ptr(), d_R, w2.data_ptr(), 1, 0,
                                                    got[i].data_ptr(), status.data_ptr(), st))
        torch.cuda.synchronize()

    t = threading.Thread(target=run)
    t.start()
    t.join()
    assert rc == [0] * n_w and int(status.item()) == 0
    ref = (torch.nn.functional.silu(z.double() @ w1.double().transpose(1, 2)) @ w2.double())[..., 0]
    # the kernels' fast exponential and division (1e-6 relative), fp32 sums over 64 terms of order one
    assert float((got.double() - ref).abs().max()) <= 1e-4 * float(ref.abs().max())
