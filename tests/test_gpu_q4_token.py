"""One token over a 4-bit cache at the edges of its kernel: groups of one to more than eight query heads, in blocks of eight and of
sixteen, caches that end inside and at the edge of a warp's 16 keys, of a tile of 64 and of a split, units in and out of
temporal order."""

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _hidden(n, D, seed):
    g = np.random.default_rng(7400 + seed)
    return W.to_bf16_grid(g.standard_normal((n, D)).astype(np.float32))


@pytest.mark.parametrize("h,hk,d", [(4, 4, 96), (8, 2, 128), (8, 1, 64), (9, 1, 128), (17, 1, 96)])
@pytest.mark.parametrize("first", [0, 1, 15, 16, 63, 64, 65, 130, 383])
def test_one_token_over_a_4_bit_cache(h, hk, d, first):
    from parity_util import lockstep_chunk, make_pair
    sh = W.LayerShape(d_model=96, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=64, rope_theta=500000.0, kv_dtype=1)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 82), budget=700, chunk=400, n_stab=16)
    if first:
        ora.prefill_chunk(_hidden(first, 96, 1), 0)
    lockstep_chunk(ora, gpu, _hidden(1, 96, 60 + first), 1, what=f"{h} {hk} {d} {first}+1")
    gpu.destroy()


@pytest.mark.parametrize("h,hk,d", [(4, 4, 96), (8, 2, 128), (8, 2, 64)])
def test_tokens_after_an_eviction(h, hk, d):
    """Slots out of temporal order: each key is rotated at its rank."""
    import torch
    from paper_2410_01805_b200 import LocretLayer
    from parity_util import bf16_dev, check_attention
    from oracle import locret_oracle as O
    sh = W.LayerShape(d_model=96, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=64, rope_theta=500000.0, kv_dtype=1)
    wts = W.layer_weights(sh, 0, seed=W.BASE_SEED + 83)
    gpu = LocretLayer(sh, *(bf16_dev(a) for a in wts), 200, 150, 8, reserve=8)
    out = torch.zeros((150, h * d), dtype=torch.bfloat16, device="cuda")
    for c in range(2):
        gpu.prefill_chunk(bf16_dev(_hidden(150, 96, c)), out, 0)
    # in temporal order: what the oracle continues from
    st = {k: v.astype(np.float64) if getattr(v, "dtype", None) in (np.float32, np.float16) else v for k, v in gpu.export_state().items()}
    ora = O.OracleLayer(sh, *wts, 200, 150, 8, mirror=True)
    ora.want_flip_sens = True
    ora.import_state(st)
    for t in range(3):
        x = _hidden(1, 96, 70 + t)
        gpu.prefill_chunk(bf16_dev(x), out[:1], O.NO_EVICT)
        ref = ora.prefill_chunk(x, O.NO_EVICT)
        check_attention(out[:1].float().cpu().numpy().astype(np.float64), ref, f"token {t}", ora.last_abs_out, ora.last_flip_sens)
    assert gpu.sync_status() == 0
    gpu.destroy()


@pytest.mark.parametrize("h,hk,d,first", [(288, 32, 64, 1987), (144, 16, 96, 3584), (80, 8, 128, 7200)])
def test_one_token_in_blocks_of_sixteen_heads(h, hk, d, first):
    """More than 6 * 148 tiles of 64 units, the last one with a few, in more blocks of eight than fit the GPU."""
    from parity_util import lockstep_chunk, make_pair
    sh = W.LayerShape(d_model=64, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=8, rope_theta=500000.0, kv_dtype=1)
    ora, gpu = make_pair(sh, W.layer_weights(sh, 0, seed=W.BASE_SEED + 84), budget=8000, chunk=first, n_stab=16)
    ora.prefill_chunk(_hidden(first, 64, 1), 0, rows=[0])
    lockstep_chunk(ora, gpu, _hidden(1, 64, 60 + first), 1, what=f"{h} {hk} {d} {first}+1")
    gpu.destroy()


@pytest.mark.parametrize("g,d", [(16, 128), (9, 96), (17, 128)])
def test_a_stack_in_blocks_of_sixteen_equals_layers_in_blocks_of_eight(g, d):
    """Eight layers in one launch have enough tiles, one alone has not; the sums are the same."""
    import torch
    from paper_2410_01805_b200 import LayerStack, LocretLayer
    from parity_util import bf16_dev
    sh = W.LayerShape(d_model=64, n_q_heads=2 * g, n_kv_heads=2, head_dim=d, d_retain=8, rope_theta=500000.0, kv_dtype=1)
    runs = []
    for stack in (True, False):
        layers = [LocretLayer(sh, *(bf16_dev(a) for a in W.layer_weights(sh, i, seed=W.BASE_SEED + 85)), 4000, 1800, 16) for i in range(8)]
        big = torch.zeros((1800, 2 * g * d), dtype=torch.bfloat16, device="cuda")
        for c in range(2):
            for L in layers:
                L.prefill_chunk(bf16_dev(_hidden(1800, 64, c)), big, 0)
        outs = torch.zeros((3, 8, 2 * g * d), dtype=torch.bfloat16, device="cuda")
        for t in range(3):
            x = bf16_dev(_hidden(1, 64, 90 + t))
            if stack:
                LayerStack(layers).decode_step(x, outs[t], out_stride=2 * g * d)
            else:
                for i, L in enumerate(layers):
                    L.decode_step(x, outs[t, i])
        assert all(L.sync_status() == 0 for L in layers)
        runs.append(outs.cpu())
        for L in layers:
            L.destroy()
    assert torch.equal(*runs)
