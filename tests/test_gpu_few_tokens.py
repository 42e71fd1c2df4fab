"""Steps of a few tokens: the projections that divide K over a cluster and the attention that divides the
key tiles, at the edges of their token tiles (16, 32, 64, 128, two tiles of 128, the wide GEMM), query
tiles and key tiles, with clusters of one to eight and shares that lie behind the causal boundary."""

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# (h, hk, d, D, d_R): K of 2048 is divided by eight, of 512 by two, of 128 not at all; 96 rows of W1 are less than a tile
SHAPES = [(4, 2, 64, 2048, 256), (3, 3, 96, 512, 96), (8, 2, 128, 128, 160)]


def _hidden(n, D, seed):
    g = np.random.default_rng(7000 + seed)
    return W.to_bf16_grid(g.standard_normal((n, D)).astype(np.float32))


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("first", [0, 5, 700])   # cached units before the step
def test_layer_steps_of_few_tokens(dims, first):
    from parity_util import lockstep_chunk, make_pair
    h, hk, d, D, dR = dims
    sh = W.LayerShape(d_model=D, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=dR, rope_theta=500000.0)
    wts = W.layer_weights(sh, 0, seed=W.BASE_SEED + 71)
    for n_tok in (2, 16, 17, 33, 64, 65, 128, 129, 257):
        ora, gpu = make_pair(sh, wts, budget=1024, chunk=max(300, first), n_stab=16)
        if first:
            ora.prefill_chunk(_hidden(first, D, 1), 0)
        lockstep_chunk(ora, gpu, _hidden(n_tok, D, n_tok), 1, what=f"{dims} {first}+{n_tok}")
        gpu.destroy()


@pytest.mark.parametrize("n_tok", [1, 2, 31, 64, 129, 257])
def test_block_steps_of_few_tokens(n_tok):
    from test_gpu_block import block_pair, lockstep_block
    sh = W.LayerShape(d_model=512, n_q_heads=4, n_kv_heads=2, head_dim=128, d_retain=64, rope_theta=500000.0, d_ff=640)
    ora, gpu = block_pair(sh, 41, budget=700, chunk=300, n_stab=16)
    ora.attn.prefill_chunk(_hidden(200, 512, 2), 0)
    lockstep_block(ora, gpu, _hidden(n_tok, 512, n_tok), 1, f"block, {n_tok} tokens")
    gpu.destroy()


@pytest.mark.parametrize("kv_dtype,n_tok", [(0, 129), (0, 256), (0, 257), (1, 300), (1, 512), (1, 513)])
def test_retaining_head_of_a_long_k(kv_dtype, n_tok):
    """K of twelve times d_model: beyond 128 tokens this path up to 256, with a 4-bit cache up to 512, and attention
    undivided beside its 128 CTAs."""
    from parity_util import lockstep_chunk, make_pair
    sh = W.LayerShape(d_model=128, n_q_heads=8, n_kv_heads=2, head_dim=128, d_retain=1024, rope_theta=500000.0, kv_dtype=kv_dtype)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 72), budget=1400, chunk=700, n_stab=16)
    ora.prefill_chunk(_hidden(700, 128, 1), 0)
    lockstep_chunk(ora, gpu, _hidden(n_tok, 128, n_tok), 1, what=f"{kv_dtype} 700+{n_tok}")
    gpu.destroy()


@pytest.mark.parametrize("kv_dtype", [0, 1])
@pytest.mark.parametrize("D", [4096, 4608])   # the last width whose layers share a launch, and one beyond
def test_one_token_of_a_wide_model(D, kv_dtype):
    from parity_util import lockstep_chunk, make_pair
    sh = W.LayerShape(d_model=D, n_q_heads=4, n_kv_heads=2, head_dim=64, d_retain=96, rope_theta=500000.0, kv_dtype=kv_dtype)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 73), budget=200, chunk=100, n_stab=16)
    ora.prefill_chunk(_hidden(90, D, 1), 0)
    for t in range(2):
        lockstep_chunk(ora, gpu, _hidden(1, D, 60 + t), 1, what=f"{D} token {t}")
    gpu.destroy()
