"""Evictions of one-token steps at the sizes where their work divides differently: rows of a block in one and in several
passes, remainders of head_dim 96 (85 rows a pass) and of a block's share, the smallest cache, and both sides of the rule that
takes the selection and the gather in one launch or in two.  Every array that an eviction rewrites is compared: token ids, scores,
K, V and, through the attention of the step after it, the rotated keys."""

import numpy as np
import pytest
import torch

import workloads as W
from oracle import locret_oracle as O

pytestmark = pytest.mark.gpu

# Rounding to bf16 of the output and of the probabilities: at most 2^-9 of each element, and of each term of a sum whose signs are
# random; a few stored elements one bf16 step apart.  Together below 2^-8 of the output's norm; twice that.
REL_TOL = 2.0 ** -7


def _attention_with_stale_keys(ora, x, gone_rank, share):
    """The oracle's attention of the next token when `share` of the units behind the last evicted one had kept their rotation."""
    h, hk, d = ora.h, ora.hk, ora.d
    q, k, v = O.split_qkv(ora._r(O.project_qkv(np.asarray(x, np.float64), ora.w_qkv, h, hk, d)), h, hk, d)
    pos = np.broadcast_to(np.arange(ora.len), (hk, ora.len)).copy()
    for m in range(hk):
        pos[m] += (np.arange(ora.len) >= gone_rank[m]) & (np.arange(ora.len) % share == share - 1)
    keys = ora._r(O.rope(ora.K, pos, ora.s.rope_theta))
    at = np.full((1, 1), ora.len)
    return O.attention_rows(ora._r(O.rope(q, at, ora.s.rope_theta)), keys, ora.V, ora._r(O.rope(k, at, ora.s.rope_theta)), v, ora.g)


@pytest.mark.parametrize("d,heads,budget,n_stab,n_prefix,first", [
    (128, (8, 8), 2401, 20, 0, [1250, 1250]),
    (96, (8, 8), 3170, 0, 5, [1600, 1600]),
    (64, (4, 2), 1, 0, 0, [1]),
    (64, (2, 2), 300, 300, 0, [200, 200]),       # nothing but the oldest unit competes: all ranks move
    (128, (1, 1), 9400, 20, 0, [4800, 4800]),    # 147 blocks, one launch
    (128, (1, 1), 9500, 20, 0, [4800, 4800]),    # 149 blocks, two launches
    (128, (8, 8), 8193, 20, 0, [4200, 4200]),    # more than 2^23 elements of keys, two launches
])
def test_evictions_of_one_unit(d, heads, budget, n_stab, n_prefix, first):
    from parity_util import FLIP_FRACTION, bf16_dev, make_pair
    from test_gpu_free_running import _hand_scored_layer
    h, hk = heads
    sh, wts = _hand_scored_layer(h, hk, d, 64, seed=d)
    ora, gpu = make_pair(sh, wts, budget, max(first), n_stab)
    ora.want_flip_sens = False
    if n_prefix:
        ora.set_protected_prefix(n_prefix)
        gpu.set_protected_prefix(n_prefix)
    g = np.random.default_rng(700 + d + n_stab)

    def hidden(n_tok):
        x = W.to_bf16_grid(g.standard_normal((n_tok, 64)).astype(np.float32))
        x[:, :hk] = g.integers(-2, 4, size=(n_tok, hk)).astype(np.float32)
        return x

    for n_tok in first:
        x = hidden(n_tok)
        gpu.prefill_chunk(bf16_dev(x), torch.zeros((n_tok, h * d), dtype=torch.bfloat16, device="cuda"), 0)
        ora.prefill_chunk(x, 0, rows=[0])
    out = torch.zeros((1, h * d), dtype=torch.bfloat16, device="cuda")
    gone_rank = None
    for t in range(6):
        x = hidden(1)
        before = gpu.compaction_counters
        stale = _attention_with_stale_keys(ora, x, gone_rank, 2) if gone_rank is not None and min(gone_rank) < budget // 2 else None
        gpu.prefill_chunk(bf16_dev(x), out, 0)
        ref = ora.prefill_chunk(x, 0)
        got = out.float().cpu().numpy().astype(np.float64)
        err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert err < REL_TOL, f"step {t}: attention off by {err:.3g} of its norm"
        if stale is not None and budget > 1:   # (what the bound is worth: half of the keys at their old positions)
            assert np.linalg.norm(stale - ref) / np.linalg.norm(ref) > 1.5 * REL_TOL
        st = gpu.export_state()
        assert np.array_equal(st["T"], ora.T), f"step {t}: retained token ids differ"
        assert np.array_equal(st["S"].astype(np.float64), ora.S), f"step {t}: scores differ"
        for name in ("K", "V"):
            diff = np.abs(st[name] - getattr(ora, name))
            assert np.all(diff <= np.abs(getattr(ora, name)) * 2.0 ** -7 + 1e-6), f"step {t}: {name} differs"
            assert np.mean(diff != 0) < FLIP_FRACTION
        # the last unit moves into the freed slot, unless it is the one that goes; every unit behind that one is rotated again
        gone_rank = [int(np.setdiff1d(np.arange(budget + 1), ora.last_keep[m])[0]) for m in range(hk)]
        moved, rotated = (b - a for a, b in zip(before, gpu.compaction_counters))
        assert moved == sum(r != budget for r in gone_rank) and rotated == sum(budget - r for r in gone_rank)
    assert gpu.sync_status() == 0
    gpu.destroy()
