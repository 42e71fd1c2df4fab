"""One-token steps that evict one unit each (a stream without an end): the retained set, ranks and scores stay the
oracle's, with ties, with everything but one unit protected, with a protected prefix, after larger evictions, and with
more candidates than one block has threads."""

import numpy as np
import pytest
import torch

import workloads as W
from oracle import locret_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,budget,n_stab,n_prefix,first", [
    (64, (4, 2), 150, 20, 0, [96, 54]),          # exactly full
    (128, (8, 2), 150, 0, 0, [96, 96, 41]),      # slots out of temporal order, nothing protected
    (96, (3, 3), 150, 150, 0, [96, 96]),         # all but the oldest unit protected
    (64, (4, 1), 150, 20, 129, [96, 96]),        # one retained unit competes with the one that leaves the stabilizers
    (64, (4, 2), 1100, 30, 3, [600, 600, 7]),    # more candidates than threads
])
def test_one_unit_evictions(d, heads, budget, n_stab, n_prefix, first):
    from parity_util import bf16_dev, make_pair
    from test_gpu_free_running import _hand_scored_layer
    h, hk = heads
    sh, wts = _hand_scored_layer(h, hk, d, 64, seed=d)
    ora, gpu = make_pair(sh, wts, budget, max(first), n_stab)
    if n_prefix:
        ora.set_protected_prefix(n_prefix)
        gpu.set_protected_prefix(n_prefix)
    g = np.random.default_rng(900 + d + n_stab)

    def step(n_tok, flags=0):
        x = W.to_bf16_grid(g.standard_normal((n_tok, 64)).astype(np.float32))
        x[:, :hk] = g.integers(-2, 4, size=(n_tok, hk)).astype(np.float32)   # many ties (below 0: score 0)
        gpu.prefill_chunk(bf16_dev(x), torch.zeros((n_tok, h * d), dtype=torch.bfloat16, device="cuda"), flags)
        ora.prefill_chunk(x, flags)

    for n_tok in first:
        step(n_tok)
    for t in range(24):
        before = gpu.compaction_counters
        step(1, O.LAST_CHUNK if t == 20 else 0)
        st = gpu.export_state()
        assert np.array_equal(st["T"], ora.T), f"step {t}: retained token ids differ"
        assert np.array_equal(st["S"].astype(np.float64), ora.S), f"step {t}: scores differ"
        moved, rotated = (b - a for a, b in zip(before, gpu.compaction_counters))
        assert 0 <= moved <= hk and moved <= rotated <= hk * budget
    assert gpu.sync_status() == 0
    gpu.destroy()
