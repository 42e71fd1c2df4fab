"""The sums of the one-token projection are rounded fp32 sums: what is left of sums that cancel is their rounding error, and it
has no sign in common.  (Tensor-core accumulation truncates: the same products came out 3e-8 to 4e-8 of the sum too small.)"""

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _cancelling(D, n_cols, seed):
    """x, w with non-negative products but for three that take their sum away, all but its last bits."""
    g = np.random.default_rng(seed)
    x = W.to_bf16_grid(np.abs(g.standard_normal(D)).astype(np.float32))
    w = W.to_bf16_grid((np.abs(g.standard_normal((D, n_cols))) / np.sqrt(D)).astype(np.float32))
    x[-8:] = 0
    x[-8:-5] = 1
    total = x[:-8].astype(np.float64) @ w[:-8].astype(np.float64)
    w[-8:] = 0
    rest = total.copy()
    for i in range(3):
        w[D - 8 + i] = W.to_bf16_grid((-rest).astype(np.float32))
        rest = rest + w[D - 8 + i].astype(np.float64)
    return x, w, total, rest


@pytest.mark.parametrize("D", [64, 256, 1024, 4096, 4608])
@pytest.mark.parametrize("layers", [1, 2])
def test_projection_sums_have_no_bias(D, layers):
    from paper_2410_01805_b200 import LayerStack, LocretLayer
    from parity_util import bf16_dev
    h = hk = 8
    d = 128
    sh = W.LayerShape(d_model=D, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=64, rope_theta=10000.0)
    d_in = (h + 2 * hk) * d
    x, w, total, rest = _cancelling(D, d_in, D)
    g = np.random.default_rng(1)
    w1 = bf16_dev(g.standard_normal((d_in, 64)).astype(np.float32))
    w2 = bf16_dev(g.standard_normal((64, hk)).astype(np.float32))
    gpu = [LocretLayer(sh, bf16_dev(w), w1, w2, 8, 8, 2, reserve=8) for _ in range(layers)]
    out = torch.zeros((layers, h * d), dtype=torch.bfloat16, device="cuda")
    LayerStack(gpu).decode_step(bf16_dev(x), out, out_stride=h * d)
    for L in gpu:
        st = L.export_state()
        got = np.concatenate([st["K"][:, 0], st["V"][:, 0]]).reshape(-1).astype(np.float64)
        err = (got - rest[h * d:]) / total[h * d:]
        # At most 2^-24 of a partial sum per rounding, of either sign.  Those at partial sums near the total count: the last
        # steps of the tree (5) and the sums across warps (16, growing evenly: sum of squares 16 / 3); the variance of a rounding
        # is a third of its bound's square, so their rms stays below 2^-24 * sqrt((5 + 16 / 3) / 3) < 2^-23.
        bound = 6 * 2.0 ** -23 / np.sqrt(err.size)
        assert abs(err.mean()) < bound, f"D = {D}: mean error {err.mean():.3g} of the sum, bound {bound:.3g}"
        assert np.sqrt(np.mean(err ** 2)) < 2.0 ** -23
        assert L.sync_status() == 0
        L.destroy()
