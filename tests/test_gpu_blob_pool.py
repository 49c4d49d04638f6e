"""Device memory of destroyed plans is reused by later ones: results stay right, memory stays bounded, also with
plans of several sizes alive at once and on several threads."""
import threading

import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _layer(w, t, out):
    plan = tb.Plan(w)
    plan.kv_compose(t.k_pool, t.v_pool)
    plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, t.k_new, t.v_new, out, None)
    return plan


def test_results_and_memory_over_many_plans():
    ws = [wl.config(1), wl.config(2), wl.config(3, requests_override=2)]
    ts = [wl.make_tensors(w, device="cuda:0", seed=i) for i, w in enumerate(ws)]
    ref = [torch.zeros_like(t.q) for t in ts]
    # five of each alive at once: as much memory as the loop below ever holds
    keep = [_layer(w, t, o) for w, t, o in zip(ws, ts, ref) for _ in range(5)]
    torch.cuda.synchronize()
    for p in keep:
        p.destroy()
    free0 = torch.cuda.mem_get_info()[0]
    rng = np.random.default_rng(0)
    out = [torch.zeros_like(t.q) for t in ts]
    alive = []
    for _ in range(150):
        i = int(rng.integers(3))
        out[i].zero_()
        alive.append(_layer(ws[i], ts[i], out[i]))
        if len(alive) > 3:
            alive.pop(int(rng.integers(4))).destroy()          # work of the others may still be queued
        torch.cuda.synchronize()
        assert torch.equal(out[i], ref[i])
    for p in alive:
        p.destroy()
    # nothing grows from plan to plan (the driver maps small allocations 2 MB at a time)
    assert free0 - torch.cuda.mem_get_info()[0] <= 8 << 20


def test_plans_on_several_threads():
    w = wl.config(2)
    ts = [wl.make_tensors(w, device="cuda:0", seed=9) for _ in range(4)]
    outs = [torch.zeros_like(t.q) for t in ts]
    ref = torch.zeros_like(ts[0].q)
    alone = _layer(w, wl.make_tensors(w, device="cuda:0", seed=9), ref)
    torch.cuda.synchronize()
    alone.destroy()
    errors = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(10):
                    p = _layer(w, ts[k], outs[k])
                    assert p.status() == 0
                    p.destroy()
        except Exception as e:       # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors
    for o in outs:
        assert torch.equal(ref, o)


def test_plans_come_and_go_while_another_thread_captures():
    """A thread-local capture stays valid while another thread destroys an idle plan, makes one, runs it and destroys it."""
    w = wl.config(2)
    t, t2 = wl.make_tensors(w, device="cuda:0", seed=3), wl.make_tensors(w, device="cuda:0", seed=3)
    ref, out, out2 = (torch.zeros_like(t.q) for _ in range(3))
    plan, idle = _layer(w, t, ref), tb.Plan(w)
    side, errors, graph = torch.cuda.Stream(), [], torch.cuda.CUDAGraph()

    def other():
        try:
            with torch.cuda.stream(side):
                idle.destroy()
                p = _layer(w, t2, out2)
                assert p.status() == 0
                p.destroy()
        except Exception as e:       # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        plan.kv_compose(t.k_pool, t.v_pool)
        th = threading.Thread(target=other)
        th.start()
        th.join()
        plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, t.k_new, t.v_new, out, None)
    graph.replay()
    torch.cuda.synchronize()
    assert not errors, errors
    assert torch.equal(out, ref) and torch.equal(out2, ref)
    assert plan.status() == 0
    plan.destroy()
