"""A launch that CUDA refuses is the failing call's error and nobody else's."""
import ctypes

import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["compose", "attention"])
def test_a_refused_launch_is_reported_once(call):
    w = wl.config(1)
    t = wl.make_tensors(w, device="cuda:0", seed=2)
    out = torch.zeros_like(t.q)
    plan = tb.Plan(w)
    slots, which = (torch.zeros(1, dtype=torch.int32, device="cuda:0") for _ in range(2))
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.12")                   # torch's, loaded already
    stream = torch.cuda.Stream()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    # a capture ended by a wait for its own stream refuses every launch until it is closed
    assert rt.cudaStreamBeginCapture(handle, 1) == 0
    assert rt.cudaStreamSynchronize(handle) != 0
    with pytest.raises(tb.TesseraError) as e:
        if call == "compose":
            plan.kv_compose(t.k_pool, t.v_pool, stream=stream)
        else:
            plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, t.k_new, t.v_new, out, None, stream=stream)
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0 and not graph.value
    rt.cudaGetLastError()
    assert e.value.status == tb.CUDA_ERROR
    tb.rope_shift_static(w.shape, t.k_pool, slots, which, [3])
    plan.kv_compose(t.k_pool, t.v_pool)
    plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, t.k_new, t.v_new, out, None)
    assert plan.status() == 0
    plan.destroy()
