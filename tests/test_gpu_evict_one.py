"""One-token evictions in one launch where a block takes its rows in two passes (eight heads of more than 37 blocks' rows), with
the remainders of head_dim 96 (85 rows a pass) and of a block's share; and the smallest cache."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,budget,n_stab,n_prefix,first", [
    (128, (8, 8), 2401, 20, 0, [1250, 1250]),
    (96, (8, 8), 3170, 0, 5, [1600, 1600]),
    (64, (4, 2), 1, 0, 0, [1]),                  # a cache of one unit
])
def test_evictions_in_several_passes(d, heads, budget, n_stab, n_prefix, first):
    from test_gpu_stream_evict import test_one_unit_evictions
    test_one_unit_evictions(d, heads, budget, n_stab, n_prefix, first)
