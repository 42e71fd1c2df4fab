"""One call for a stack of layers puts the layers of a batch through one launch per kernel: the same bits as one call
per layer, for more layers than a batch holds, for caches of different lengths and ranks, for 4-bit caches, for
outputs that share memory and for a layer that occurs twice."""

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _hidden(n, D, seed):
    g = np.random.default_rng(8100 + seed)
    return W.to_bf16_grid(g.standard_normal((n, D)).astype(np.float32))


def _run(sh, budgets, order, use_stack, stride_rows=True, steps=3, over=None):
    from paper_2410_01805_b200 import LayerStack, LocretLayer
    from parity_util import bf16_dev
    layers = [LocretLayer(sh, *(bf16_dev(a) for a in W.layer_weights(sh, i, seed=W.BASE_SEED + 9)), b, 200, 16, reserve=16)
              for i, b in enumerate(budgets)]
    width = sh.n_q_heads * sh.head_dim
    out = torch.zeros((200, width), dtype=torch.bfloat16, device="cuda")
    for c in range(2):
        x = bf16_dev(_hidden(200, sh.d_model, c))
        for L in layers:
            L.prefill_chunk(x, out, 0)     # the smaller budgets evict: their slots are out of temporal order
    picked = [layers[i] for i in order]
    outs = torch.zeros((steps, len(picked) if stride_rows else 1, width), dtype=torch.bfloat16, device="cuda")
    stack = LayerStack(picked)
    for t in range(steps):
        x = bf16_dev(_hidden(1, sh.d_model, 50 + t))
        if over is not None:   # the input lies where layer `over` writes
            outs[t, over] = x[0]
            x = outs[t, over:over + 1]
        if use_stack:
            stack.decode_step(x, outs[t], out_stride=width if stride_rows else 0)
        else:
            for i, L in enumerate(picked):
                L.decode_step(x, outs[t, i if stride_rows else 0])
    assert all(L.sync_status() == 0 for L in layers)
    states = [dict(L.export_state(), launches=L.launch_count) for L in layers]
    got = outs.clone()
    for L in layers:
        L.destroy()
    return got, states


@pytest.mark.parametrize("d,h,hk,kw,budgets,order,stride_rows", [
    (128, 8, 2, {}, [300] * 10, range(10), True),                       # a batch of eight and one of two
    (64, 4, 2, {}, [300, 390, 150, 400], range(4), True),               # different lengths, ranks and split counts
    (96, 3, 3, dict(kv_dtype=1), [300, 350, 300], range(3), True),      # 4-bit caches
    (128, 8, 2, dict(kv_dtype=1), [300, 350, 300], range(3), True),
    (64, 64, 2, dict(rh_input=1), [300, 300], range(2), True),          # two groups of 16 heads; post-RoPE scores
    (64, 4, 2, {}, [300, 300, 300], range(3), False),                   # outputs share memory: the last layer's stay
    (64, 4, 2, {}, [300, 300], [0, 1, 0], True),                        # a layer that occurs twice
])
def test_stack_call_equals_calls_per_layer(d, h, hk, kw, budgets, order, stride_rows):
    sh = W.LayerShape(d_model=256, n_q_heads=h, n_kv_heads=hk, head_dim=d, d_retain=128, rope_theta=500000.0, **kw)
    a, sa = _run(sh, budgets, list(order), False, stride_rows)
    b, sb = _run(sh, budgets, list(order), True, stride_rows)
    assert torch.equal(a, b)
    for x, y in zip(sa, sb):
        for key in x:
            assert np.array_equal(x[key], y[key]), key


@pytest.mark.parametrize("over", [0, 1, 3])
def test_an_output_over_the_input(over):
    sh = W.LayerShape(d_model=256, n_q_heads=4, n_kv_heads=2, head_dim=64, d_retain=128, rope_theta=500000.0)
    (a, sa), (b, sb) = (_run(sh, [300] * 4, range(4), use_stack, over=over) for use_stack in (False, True))
    assert torch.equal(a, b)
    for x, y in zip(sa, sb):
        for key in x:
            assert np.array_equal(x[key], y[key]), key


@pytest.mark.parametrize("kv_dtype", [0, 1])
def test_a_captured_step_outlives_the_arrival_of_other_layers(kv_dtype):
    """A one-token step captured in a CUDA graph, more layers of the same shape on its stream, their steps, then the replay:
    the output of the same step called directly."""
    from paper_2410_01805_b200 import LayerStack, LocretLayer
    from parity_util import bf16_dev
    sh = W.LayerShape(d_model=256, n_q_heads=8, n_kv_heads=2, head_dim=128, d_retain=128, rope_theta=500000.0, kv_dtype=kv_dtype)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        def layer(i):
            return LocretLayer(sh, *(bf16_dev(a) for a in W.layer_weights(sh, i, seed=W.BASE_SEED + 9)), 300, 200, 16, reserve=16)
        x, tok = bf16_dev(_hidden(200, 256, 1)), bf16_dev(_hidden(2, 256, 2))
        out = torch.zeros((200, 1024), dtype=torch.bfloat16, device="cuda")
        outs = torch.zeros((9, 1024), dtype=torch.bfloat16, device="cuda")
        first, twin = layer(0), layer(0)
        for L in (first, twin):
            L.prefill_chunk(x, out, 0)
            L.decode_step(tok[0], outs[0])   # (the chunk's work on the second stream has been waited for)
        twin.decode_step(tok[1], outs[1])
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st, capture_error_mode="relaxed"):
            first.decode_step(tok[1], outs[0])
        others = [layer(i) for i in range(1, 8)]
        for L in others:
            L.prefill_chunk(x, out, 0)
        LayerStack(others).decode_step(tok[0], outs[2:], out_stride=1024)
        st.synchronize()
        for _ in range(2):
            outs[0] = 0
            graph.replay()
            st.synchronize()
            assert torch.equal(outs[0], outs[1])
        del graph
        for L in [first, twin] + others:
            assert L.sync_status() == 0
            L.destroy()
