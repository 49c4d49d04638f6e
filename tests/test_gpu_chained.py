"""Kernels of successive calls overlap (programmatic dependent launch): a run of layers queued without a
wait, and the same run captured in a CUDA graph, give the bits of the run that waits after every call."""
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: wl.config(1), lambda: wl.config(2), lambda: wl.config(3, requests_override=3)])
def test_queued_and_captured_layers_match_layers_with_a_wait_between(make):
    w = make()
    layers = 5
    plan = tb.Plan(w)

    def fresh():
        ts = [wl.make_tensors(w, layer=l, device="cuda:0") for l in range(layers)]
        # all layers share one pool, so that every call rewrites what the one before it read
        for t in ts[1:]:
            t.k_pool, t.v_pool = ts[0].k_pool, ts[0].v_pool
        outs = [torch.zeros(w.n_q, w.shape.num_q_heads, w.shape.head_dim, dtype=torch.bfloat16, device="cuda:0") for _ in ts]
        lses = [torch.zeros(w.n_q, w.shape.num_q_heads, dtype=torch.float32, device="cuda:0") for _ in ts]
        return ts, outs, lses

    def go(state, wait):
        for t, o, l in zip(*state):
            plan.kv_compose(t.k_pool, t.v_pool)
            wait()
            plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, t.k_new, t.v_new, o, l)
            wait()

    ref, queued, captured = fresh(), fresh(), fresh()
    go(ref, torch.cuda.synchronize)
    go(queued, lambda: None)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        go(captured, lambda: None)
    graph.replay()
    torch.cuda.synchronize()
    assert plan.status() == 0
    for other in (queued, captured):
        assert torch.equal(ref[0][0].k_pool, other[0][0].k_pool) and torch.equal(ref[0][0].v_pool, other[0][0].v_pool)
        for l in range(layers):
            assert torch.equal(ref[1][l], other[1][l]) and torch.equal(ref[2][l], other[2][l])
    plan.destroy()
