"""What creating and destroying plans does with device memory, on the CPU: the library's host sources linked with a
stand-in for the CUDA runtime (fake_cuda.cpp)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_32999_b200", "csrc")
SHAPE = wl.ModelShape(32, 8, 128, 64, 500000.0)
MB = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    """libtessera's host half over the stand-in, behind the binding's Plan."""
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    sources = [os.path.join(CSRC, f) for f in ("api.cu", "plan.cu", "blob_pool.cu")]
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                           "-I", os.path.join(cuda, "include"), "-I", CSRC, "-I", os.path.join(os.path.dirname(HERE), "include"),
                           "-x", "c++", *sources, os.path.join(HERE, "fake_cuda.cpp"), "-o", so])
    fake = ctypes.CDLL(so)
    fake.fake_reset.argtypes = fake.fake_limit.argtypes = fake.fake_host_limit.argtypes = [ctypes.c_size_t]
    fake.fake_fail_call.argtypes = [ctypes.c_long]
    fake.fake_count.argtypes, fake.fake_count.restype = [ctypes.c_char_p], ctypes.c_long
    for n in ("tessera_plan_create", "tessera_plan_destroy", "tessera_plan_get_info", "tessera_plan_status", "tessera_last_error",
              "tessera_composed_prefill_host"):
        getattr(fake, n).argtypes = getattr(tb._lib, n).argtypes
        getattr(fake, n).restype = ctypes.c_int32
    real, tb._lib = tb._lib, fake
    yield fake
    tb._lib = real


@pytest.fixture
def cuda(lib):
    lib.fake_reset(4096 * MB)
    yield lib


def _count(lib, what):
    return lib.fake_count(what.encode())


def _workload(requests, tokens, tail=64, shape=SHAPE):
    reqs = [[wl.unit(512, (r, i), recompute=()) for i in range(tokens // 512)] + [tail] for r in range(requests)]
    return wl.build_workload("memory", shape, reqs, np.random.default_rng(0))


def _plan(w):
    return tb.Plan(w, stream=0)


def test_a_block_is_used_again(cuda):
    w = _workload(1, 5120)
    _plan(w).destroy()
    n = _count(cuda, "live_bytes")
    assert 0 < n <= 192 * MB
    for _ in range(5):
        _plan(w).destroy()
        assert _count(cuda, "live_bytes") == n
    assert _count(cuda, "foreign_frees") == _count(cuda, "foreign_writes") == 0


def test_a_block_stays_with_the_context_it_came_from(cuda):
    """Made in the primary context, destroyed while another one of the same device is current: the next plan there
    must not write to it, and nothing of a live context is forgotten."""
    w = _workload(1, 5120)
    plans = [_plan(w) for _ in range(3)]
    cuda.fake_push_other_context()
    for p in plans:
        p.destroy()
    _plan(w).destroy()
    _plan(w).destroy()
    assert _count(cuda, "foreign_writes") == 0
    cuda.fake_pop_context()
    _plan(w).destroy()
    assert _count(cuda, "foreign_writes") == _count(cuda, "foreign_frees") == 0
    assert _count(cuda, "live_bytes") <= 192 * MB


def test_blocks_do_not_outlive_a_device_reset(cuda):
    w = _workload(1, 5120)
    _plan(w).destroy()
    old = _plan(w)
    cuda.fake_device_reset()
    p = _plan(w)
    assert _count(cuda, "foreign_writes") == 0
    with pytest.raises(tb.TesseraError):    # its memory went with the reset, and may be another plan's by now
        old.destroy()
    assert not old._h                       # it is gone all the same: nothing may free it a second time
    p.destroy()
    _plan(w).destroy()
    assert _count(cuda, "foreign_writes") == 0


def test_many_sizes_stay_within_the_bound(cuda):
    """More than sixteen blocks of different sizes: the oldest are given back."""
    plans = [_plan(_workload(1 + i, 512 * (1 + 3 * i), tail=16)) for i in range(24)]
    assert _count(cuda, "live_bytes") > 192 * MB
    for p in plans:
        p.destroy()
    assert _count(cuda, "live_bytes") <= 192 * MB
    assert _count(cuda, "live") <= 16 + 1
    assert _count(cuda, "foreign_frees") == 0


def test_kept_blocks_are_given_back_when_memory_runs_out(cuda):
    small, large = _workload(1, 512), _workload(4, 33000 // 512 * 512, tail=256)
    p = _plan(large)
    need = _count(cuda, "live_bytes")
    p.destroy()
    cuda.fake_reset(4096 * MB)
    alive = [_plan(small) for _ in range(12)]
    for q in alive:
        q.destroy()
    assert _count(cuda, "live_bytes") > 0
    cuda.fake_limit(need + MB // 8)
    _plan(large).destroy()                 # fits only without the kept blocks
    assert _count(cuda, "last_error") == 0


def test_destroying_a_plan_leaves_captures_of_other_threads_alone(cuda):
    """A thread-local or relaxed capture forbids waiting for the device, on any thread; freeing memory it allows."""
    w = _workload(1, 5120)
    plans = [_plan(w) for _ in range(2)]
    cuda.fake_capture_elsewhere(1)
    for p in plans:
        p.destroy()
    _plan(w).destroy()
    assert not _count(cuda, "capture_broken") and _count(cuda, "last_error") == 0


def test_a_block_is_used_again_only_when_the_device_is_idle(cuda):
    w = _workload(1, 5120)
    for _ in range(4):
        p = _plan(w)
        cuda.fake_busy(1)                  # the plan's kernels are still queued
        p.destroy()
    _plan(w).destroy()
    assert _count(cuda, "writes_while_busy") == 0


def test_a_refused_allocation_refuses_the_plan_also_beside_kept_blocks(cuda):
    w = _workload(1, 5120)
    _plan(w).destroy()
    cuda.fake_forbid_malloc(1)             # what a global capture does
    with pytest.raises(tb.TesseraError):
        _plan(w)
    cuda.fake_forbid_malloc(0)
    n = _count(cuda, "live_bytes")
    _plan(w).destroy()
    assert _count(cuda, "live_bytes") == n and _count(cuda, "foreign_frees") == 0


def test_the_largest_workspace_is_kept_for_the_next_plan(cuda):
    """Lists of one to four rounds of items, cut: the block of the largest workspace there is must not be allocated anew."""
    largest = 0
    for requests, tokens, tail, shape in [(21, 43520, 32, wl.ModelShape(64, 8, 128, 64, 500000.0)), (10, 12288, 64, SHAPE),
                                          (40, 16896, 32, wl.ModelShape(20, 4, 128, 64, 500000.0))]:
        w = _workload(requests, tokens, tail, shape)
        cuda.fake_reset(4096 * MB)
        _plan(w).destroy()
        n, kept = _count(cuda, "mallocs"), _count(cuda, "live_bytes")
        _plan(w).destroy()
        assert _count(cuda, "mallocs") == n + 1 and _count(cuda, "live_bytes") == kept      # the guard alone
        largest = max(largest, kept)
    assert 100 * MB < largest <= 192 * MB


def test_nothing_is_cut_where_the_workspace_does_not_fit(cuda):
    w = _workload(10, 12288)
    p = _plan(w)
    cut, need = p.info.n_attn_items, _count(cuda, "live_bytes")
    p.destroy()
    cuda.fake_reset(need // 2)
    p = _plan(w)
    assert p.info.n_attn_items < cut and p.info.n_attn_items == 80
    assert _count(cuda, "last_error") == 0 and _count(cuda, "foreign_writes") == 0
    p.destroy()
    cuda.fake_reset(MB // 16)              # not even the tables
    with pytest.raises(tb.TesseraError) as e:
        _plan(w)
    assert e.value.status == tb.CUDA_ERROR


def test_host_memory_running_out_is_an_error(cuda):
    """Whichever of the plan's host allocations fails - the image of the device tables is the largest - nothing throws
    through the C call, and the device keeps nothing of the plan."""
    w = _workload(2, 5120)
    _plan(w).destroy()
    live = _count(cuda, "live_bytes")
    refused = 0
    for limit in np.geomspace(64, 4 * MB, 120).astype(int).tolist():
        cuda.fake_host_limit(limit)
        try:
            _plan(w).destroy()
        except tb.TesseraError as e:
            refused += 1
            assert e.status == tb.INVALID_ARG
        finally:
            cuda.fake_host_limit(ctypes.c_size_t(-1).value)
    assert 10 < refused < 120
    assert _count(cuda, "live_bytes") == live


def test_a_host_call_that_failed_half_way_is_made_up_for_by_the_next(cuda):
    """Its streams, events and staging buffers are made by the first call; whichever of them fails, that call is
    refused and the next one finds or makes all of them."""
    w = _workload(3, 1024)
    buf = np.zeros(1 << 24, np.uint8)
    pool = (buf.ctypes.data + 255) // 256 * 256
    ptr = type("T", (), {"data_ptr": lambda self: pool})()
    for k in range(1, 40):
        p = _plan(w)
        cuda.fake_fail_call(k)
        try:
            p.composed_prefill_host(*[ptr] * 7, stream=0)
            done = True
        except tb.TesseraError as e:
            assert e.status == tb.CUDA_ERROR
            done = False
        cuda.fake_fail_call(-1)
        p.composed_prefill_host(*[ptr] * 7, stream=0)
        p.destroy()
        assert _count(cuda, "foreign_writes") == 0
        if done:
            break
    assert 10 < k < 39                     # the buffers, two streams, two events and two for each chunk


def test_staging_buffers_are_kept_for_the_next_plan(cuda):
    """A first call through host buffers allocates its guard and nothing else once a plan like it has come and gone."""
    w = _workload(3, 1024)
    buf = np.zeros(1 << 24, np.uint8)
    pool = (buf.ctypes.data + 255) // 256 * 256
    ptr = type("T", (), {"data_ptr": lambda self: pool})()
    mallocs = []
    for _ in range(4):
        p = _plan(w)
        n = _count(cuda, "mallocs")
        p.composed_prefill_host(*[ptr] * 7, stream=0)
        mallocs.append(_count(cuda, "mallocs") - n)
        p.destroy()
    assert mallocs == [2, 1, 1, 1] and _count(cuda, "foreign_writes") == 0
