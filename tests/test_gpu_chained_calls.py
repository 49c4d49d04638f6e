"""Every kind of call, queued behind one another without a wait and captured in a graph, gives the bits of the run that
waits after each call - for plans whose kernels overlap (programmatic dependent launch), alone and in turn with a plan
whose kernels do not."""
import copy

import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl
from tests.test_cut_rule import is_chained

pytestmark = pytest.mark.gpu
DEV, S8, LAYERS = "cuda:0", 1 / 32, 4


def _batch(kind):
    shape = wl.ModelShape(16, 4, 128, 32, 500000.0)
    rng = np.random.default_rng(8)
    reqs = [[5] + [wl.unit(130 + 9 * i, (r, i), cached=i != 1 or kind != "extend", stride=i % 2, recompute=(0, 7)) for i in range(4)] + [40 + r]
            for r in range(3)]
    w = wl.build_workload(kind, shape, reqs, rng)
    if kind in ("fp8", "key8", "store"):
        w.num_source_pages = w.num_pool_pages
    if kind == "extend":                   # the missed unit of every request is captured into pages behind the pool
        off, pages, page = [0], [], w.num_pool_pages
        for u in range(len(w.unit_len)):
            if w.unit_page_off[u + 1] == w.unit_page_off[u]:
                n = -(-int(w.unit_len[u]) // shape.page_size)
                pages += range(page, page + n)
                page += n
            off.append(len(pages))
        w.unit_retain_page_off, w.unit_retain_pages, w.num_pool_pages = np.array(off, np.int32), np.array(pages, np.int32), page
    return w


class _State:
    """Layers with tensors of their own over one pool, so that every call rewrites what the one before it read."""

    def __init__(self, w, kind):
        ts = [wl.make_tensors(w, layer=l, device=DEV) for l in range(LAYERS)]
        self.kind = kind
        self.k, self.v = ts[0].k_pool, ts[0].v_pool
        self.src = [(t.k_pool.clone(), t.v_pool.clone()) if kind in ("fp8", "key8", "store") else None for t in ts]
        if kind == "fp8":
            self.src = [tuple((x.float() / S8).to(torch.float8_e4m3fn).view(torch.uint8) for x in p) for p in self.src]
        if kind in ("key8", "store"):
            self.k8, self.v8 = (torch.zeros(self.k.shape, dtype=torch.uint8, device=DEV) for _ in range(2))
        self.q, self.k_new, self.v_new = [t.q for t in ts], [t.k_new for t in ts], [t.v_new for t in ts]
        self.out = [torch.zeros_like(t.q) for t in ts]
        self.lse = [torch.zeros(t.q.shape[:2], dtype=torch.float32, device=DEV) for t in ts]

    def layer(self, plan, l, wait):
        k, v, src, q, kn, vn, out, lse = self.k, self.v, self.src[l], self.q[l], self.k_new[l], self.v_new[l], self.out[l], self.lse[l]
        if self.kind == "plain":
            calls = [lambda: plan.kv_compose(k, v), lambda: plan.partial_prefill_attn(k, v, q, kn, vn, out, lse)]
        elif self.kind == "unfused":
            calls = [lambda: plan.kv_compose(k, v, fuse_rope=False), lambda: plan.rope_shift(k), lambda: plan.rope_fresh(q, kn),
                     lambda: plan.partial_prefill_attn(k, v, q, kn, vn, out, lse)]
        elif self.kind == "extend":
            calls = [lambda: plan.kv_compose(k, v), lambda: plan.extend_write(k, v, q, kn, vn, k, v),
                     lambda: plan.partial_prefill_attn(k, v, q, None, None, out, lse)]
        elif self.kind == "fp8":
            calls = [lambda: plan.kv_compose_from_fp8(*src, S8, S8, k, v), lambda: plan.partial_prefill_attn(k, v, q, kn, vn, out, lse)]
        elif self.kind == "key8":
            calls = [lambda: plan.kv_compose_k8(*src, self.k8, v, S8),
                     lambda: plan.partial_prefill_attn_k8(self.k8, S8, v, q, S8, kn, vn, out, lse)]
        else:
            calls = [lambda: plan.kv_compose_from(*src, k, v), lambda: plan.kv_retain_fp8(k, v, self.k8, self.v8, S8, S8)]
        for call in calls:
            call()
            wait()

    def bits(self):
        all_ = [self.k, self.v, *self.q, *self.k_new, *self.out, *self.lse] + ([self.k8, self.v8] if self.kind in ("key8", "store") else [])
        return [x.view(torch.uint8) for x in all_]


@pytest.mark.parametrize("beside", [False, True])
@pytest.mark.parametrize("kind", ["plain", "unfused", "extend", "fp8", "key8", "store"])
def test_queued_and_captured_calls_match_calls_with_a_wait_between(kind, beside):
    w, wide = _batch(kind), wl.config(4, requests_override=1)
    assert is_chained(w) and not is_chained(wide)
    plan, wide_plan = tb.Plan(w), tb.Plan(wide) if beside else None

    def fresh():
        torch.manual_seed(0)
        return _State(w, kind), _State(wide, "plain") if beside else None

    def go(states, wait):
        for l in range(LAYERS):
            states[0].layer(plan, l, wait)
            if beside:
                states[1].layer(wide_plan, l, wait)

    ref, queued = fresh(), fresh()
    go(ref, torch.cuda.synchronize)
    go(queued, lambda: None)
    torch.cuda.synchronize()
    captured = fresh()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        go(captured, lambda: None)
    graph.replay()
    torch.cuda.synchronize()
    assert plan.status() == 0 and (not beside or wide_plan.status() == 0)
    for other in (queued, captured):
        for a, b in zip(ref, other):
            if a is not None:
                for i, (x, y) in enumerate(zip(a.bits(), b.bits())):
                    assert torch.equal(x, y), (kind, i)
    plan.destroy()
    if beside:
        wide_plan.destroy()
