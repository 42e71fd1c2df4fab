"""The wide GEMMs on pairs of CTAs (256-row tiles): whole and half-empty last tiles, one tile of a pair and several in one and in more
than one wave, column remainders, every epilogue: projection with RoPE for the three head sizes, retaining head, residual, gated
FFN, pre-activations and gradients."""

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _hidden(n, D, seed):
    g = np.random.default_rng(7300 + seed)
    return W.to_bf16_grid(g.standard_normal((n, D)).astype(np.float32))


# (h, hk, d, D, d_R): a projection of 4 x 256 and of 3 x 192 columns, and one whose last tile is half empty
@pytest.mark.parametrize("dims", [(8, 4, 64, 256, 256), (2, 2, 96, 192, 512), (5, 1, 128, 320, 128)])
@pytest.mark.parametrize("n_tok", [513, 640, 641, 768, 1000])
def test_layer_steps(dims, n_tok):
    from parity_util import lockstep_chunk, make_pair
    h, hk, d, D, dR = dims
    sh = W.LayerShape(d_model=D, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=dR, rope_theta=500000.0)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 81), budget=1200, chunk=1000, n_stab=16)
    ora.prefill_chunk(_hidden(70, D, 1), 0)
    lockstep_chunk(ora, gpu, _hidden(n_tok, D, n_tok), 1, what=f"{dims} {n_tok}")
    gpu.destroy()


# more than 74 pair tiles in no more waves than single CTAs take: 17 column tiles of 256 (of 192) x 6 pairs of row blocks, of which the
# last is half empty, or full but for a few rows
@pytest.mark.parametrize("dims", [(30, 2, 128, 64, 64), (64, 2, 64, 64, 64), (30, 2, 96, 64, 64)])
@pytest.mark.parametrize("n_tok", [1358, 1530])
def test_projections_of_several_waves(dims, n_tok):
    from parity_util import lockstep_chunk, make_pair
    h, hk, d, D, dR = dims
    sh = W.LayerShape(d_model=D, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=dR, rope_theta=500000.0)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 86), budget=1700, chunk=1536, n_stab=16)
    ora.prefill_chunk(_hidden(70, D, 1), 0)
    rows = [0, 127, 128, 255, 256, 1151, 1152, 1279, 1280, n_tok - 1]
    lockstep_chunk(ora, gpu, _hidden(n_tok, D, n_tok), 1, rows=rows, what=f"{dims} {n_tok}")
    gpu.destroy()


@pytest.mark.parametrize("n_tok", [530, 769])
def test_block_steps(n_tok):
    from test_gpu_block import block_pair, lockstep_block
    sh = W.LayerShape(d_model=512, n_q_heads=4, n_kv_heads=2, head_dim=128, d_retain=64, rope_theta=500000.0, d_ff=640)
    ora, gpu = block_pair(sh, 43, budget=900, chunk=800, n_stab=16)
    lockstep_block(ora, gpu, _hidden(n_tok, 512, n_tok), 1, f"block, {n_tok} tokens")
    gpu.destroy()


# the last: 39 row blocks x 4 column tiles of pre-activations, a second wave whose last pair tile is half empty
@pytest.mark.parametrize("n,d_in,d_R,hk", [(192, 320, 256, 8), (640, 448, 512, 4), (4928, 128, 1024, 2)])
def test_loss_and_gradients(n, d_in, d_R, hk):
    from test_gpu_train import test_loss_and_gradients_match_the_oracle
    test_loss_and_gradients_match_the_oracle(n, d_in, d_R, hk)
