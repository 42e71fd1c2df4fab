"""Eq. 1 on tcgen05 at the edges of its arithmetic: scores that are NaN, infinite or far below zero, in one key tile or one
share of the keys, and what must not reach an output: the values of masked keys and of slots behind the cache's end."""

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _layer(d, h=4, hk=2, D=128, cap=2000, wqkv=None, theta=1e30, **kw):
    """rope_theta 1e30: the last pair of a head does not turn, so a test can fix its scores by hand."""
    from paper_2410_01805_b200 import LocretLayer
    from parity_util import bf16_dev
    sh = W.LayerShape(d_model=D, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=64, rope_theta=theta, **kw)
    w = [np.array(a) for a in W.layer_weights(sh, 0, seed=W.BASE_SEED + 41)]
    if wqkv is not None:
        w[0] = wqkv(w[0], sh)
    return sh, LocretLayer(sh, *(bf16_dev(a) for a in w), cap - 300, 300, 0)


def _import(gpu, sh, K, V):
    hk, n = K.shape[:2]
    gpu.import_state(K, V, np.zeros((hk, n), np.float32), np.broadcast_to(np.arange(n), (hk, n)).copy(), n)


def _step(gpu, sh, x, flags=1):
    from parity_util import bf16_dev
    out = torch.zeros((x.shape[0], sh.n_q_heads * sh.head_dim), dtype=torch.bfloat16, device="cuda")
    gpu.prefill_chunk(bf16_dev(x), out, flags)
    return out.float().cpu().numpy().reshape(x.shape[0], sh.n_q_heads, sh.head_dim)


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", [(0, 128), (1024, 1025), (640, 700)])
def test_nan_scores_are_not_lost(d, bad, where):
    """Keys of KV head 0 whose scores are NaN (a NaN key, or an infinite one against both signs of a query): every row that
    sees one is NaN in that head's group, however the keys are divided, and the other group is not."""
    g = np.random.default_rng(11)
    sh, gpu = _layer(d)
    for n_tok in (2, 5, 70, 200):   # (the first key tile is a share of its own where nine tiles are divided in five or more)
        K = W.to_bf16_grid(g.standard_normal((2, 1025, d)).astype(np.float32))
        V = W.to_bf16_grid(g.standard_normal((2, 1025, d)).astype(np.float32))
        K[0, where[0]:where[1]] = bad
        _import(gpu, sh, K, V)
        out = _step(gpu, sh, W.to_bf16_grid(g.standard_normal((n_tok, 128)).astype(np.float32)))
        assert np.isnan(out[:, :2]).all(), n_tok
        assert np.isfinite(out[:, 2:]).all(), n_tok
    assert gpu.sync_status() == 0
    gpu.destroy()


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("n_tok,cached", [(2, 1024), (40, 700), (150, 1500), (2, 100)])
def test_scores_far_below_zero(d, n_tok, cached):
    """Every score of a row is the same -1e36: the output is the mean of the values it sees."""
    g = np.random.default_rng(12)
    i = d // 2 - 1   # the pair that does not turn

    def weights(w, sh):
        w = np.zeros_like(w)
        for hd in range(sh.n_q_heads):
            w[0, hd * d + i] = 1.0
        for m in range(sh.n_kv_heads):
            w[0, (sh.n_q_heads + m) * d + i] = -1.0
            w[1:, (sh.n_q_heads + sh.n_kv_heads + m) * d:][:, :d] = W.to_bf16_grid(
                (g.standard_normal((w.shape[0] - 1, d)) / 8).astype(np.float32))
        return w

    sh, gpu = _layer(d, wqkv=weights)
    x = W.to_bf16_grid(g.standard_normal((n_tok, 128)).astype(np.float32))
    x[:, 0] = 2.0 ** 60
    K = np.zeros((2, cached, d), np.float32)
    K[:, :, i] = -(2.0 ** 60)
    V = W.to_bf16_grid((1 + g.standard_normal((2, cached, d))).astype(np.float32))
    _import(gpu, sh, K, V)
    out = _step(gpu, sh, x)
    st = gpu.export_state()
    allV = st["V"].astype(np.float64)
    csum = np.cumsum(allV, axis=1)
    for r in range(n_tok):
        ref = np.repeat(csum[:, cached + r] / (cached + r + 1), 2, axis=0)
        # P is exactly one in every key: fp32 sums and one bf16 rounding of the result
        tol = 2.0 ** -8 * np.abs(ref) + 2.0 ** -12 * np.abs(allV[:, :cached + r + 1]).mean()
        assert (np.abs(out[r] - ref) <= tol).all(), (r, np.abs(out[r] - ref).max())
    assert gpu.sync_status() == 0
    gpu.destroy()


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("n_tok,cached", [(40, 0), (40, 900), (200, 0), (280, 1500)])
def test_masked_values_weigh_nothing(d, n_tok, cached):
    """The values of a later token, however large, leave the rows before it as they are, bit for bit."""
    g = np.random.default_rng(13)

    def weights(w, sh):   # column 0 of the input reaches the values alone
        w[0] = 0.0
        w[0, (sh.n_q_heads + sh.n_kv_heads) * d:] = 1.0
        return w

    sh, gpu = _layer(d, wqkv=weights, theta=10000.0)
    x = W.to_bf16_grid(g.standard_normal((n_tok, 128)).astype(np.float32))
    K, V = (W.to_bf16_grid(g.standard_normal((2, max(cached, 1), d)).astype(np.float32)) for _ in range(2))
    outs = []
    for big in (0.0, 2.0 ** 126):
        x[n_tok // 2:, 0] = big
        if cached:
            _import(gpu, sh, K, V)
        else:
            gpu.reset()
        outs.append(_step(gpu, sh, x)[:n_tok // 2])
    assert np.array_equal(outs[0], outs[1])
    assert gpu.sync_status() == 0
    gpu.destroy()


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("kind", ["bf16", "int4", "heads"])
def test_slots_behind_the_end_do_not_reach_an_output(d, kind):
    """A request with NaN inputs, a reset, then a short request: the bits of a layer that never saw the first."""
    g = np.random.default_rng(14)
    kw = dict(kv_dtype=1) if kind == "int4" else {}
    sh, used = _layer(d, theta=10000.0, **kw)
    x = W.to_bf16_grid(g.standard_normal((270, 128)).astype(np.float32))
    poison = np.full((300, 128), np.nan, np.float32)
    for sizes in ([1, 20, 1], [2], [63], [64, 1], [130], [200, 45], [270]):
        outs = []
        for gpu in (used, _layer(d, theta=10000.0, **kw)[1]):
            if kind == "heads":
                gpu.reset()
                gpu.set_head_budgets([1600, 1500])
            if gpu is used:
                _step(gpu, sh, poison)
                gpu.reset()
            t = 0
            for n in sizes:
                outs.append(_step(gpu, sh, x[t:t + n]))
                t += n
            assert gpu.sync_status() == 0
        half = len(sizes)
        for a, b in zip(outs[:half], outs[half:]):
            assert np.isfinite(b).all() and np.array_equal(a, b), sizes
