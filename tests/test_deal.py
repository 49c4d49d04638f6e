"""How the planner deals the attention's work list out to the thread blocks, on the CPU."""
import ctypes
import heapq
import os
import random
import subprocess

import numpy as np
import pytest

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_32999_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    """libtessera's host half with a window on its plans, behind the binding's Plan."""
    so = str(tmp_path_factory.mktemp("view") / "libview.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    sources = [os.path.join(CSRC, f) for f in ("api.cu", "plan.cu", "blob_pool.cu")]
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                           "-I", os.path.join(cuda, "include"), "-I", CSRC, "-I", os.path.join(os.path.dirname(HERE), "include"),
                           "-x", "c++", *sources, os.path.join(HERE, "fake_cuda.cpp"), os.path.join(HERE, "plan_view.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    for n in ("tessera_plan_create", "tessera_plan_destroy", "tessera_plan_get_info", "tessera_last_error"):
        getattr(lib, n).argtypes, getattr(lib, n).restype = getattr(tb._lib, n).argtypes, ctypes.c_int32
    lib.view_work.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_int]
    lib.view_tile_steps.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    lib.view_chunks.argtypes = [ctypes.c_void_p]
    lib.view_grid.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    real, tb._lib = tb._lib, lib
    yield lib
    tb._lib = real


class Deal:
    """The lists of one plan: items, their modelled cycles, and what every thread block is handed."""

    def __init__(self, view, w):
        plan = tb.Plan(w, host_only=True)
        n = view.view_work(plan._h, 0, None, 0)
        self.work, self.items = np.zeros((n, 12), np.int32), np.zeros((view.view_work(plan._h, 1, None, 0), 12), np.int32)
        view.view_work(plan._h, 0, self.work.ctypes.data, n)
        view.view_work(plan._h, 1, self.items.ctypes.data, len(self.items))
        tiles = np.zeros(max(1, view.view_tile_steps(plan._h, None, 0)), np.int32)
        view.view_tile_steps(plan._h, tiles.ctypes.data, len(tiles))
        self.row_bytes, self.kv_heads, self.tokens = w.shape.head_dim * 4, w.shape.num_kv_heads, int(w.seq_len.sum())
        plan.destroy()
        self.grid = min(n, SMS)
        self.mine = [[] for _ in range(self.grid)]              # the kernel's walk
        for i in range(n):
            k, j = divmod(i, self.grid)
            self.mine[self.grid - 1 - j if k & 1 else j].append(i)
        self.real = self.work[:, 0] >= 0
        self.cycles = np.array([self._cycles(x, tiles) if x[0] >= 0 else 0 for x in self.work], np.int64)
        self.mean_steps = (self.work[self.real, 4] - self.work[self.real, 3]).mean()

    @staticmethod
    def _cycles(x, tiles):
        a, b = min(x[4], tiles[x[0]]) - x[3], min(x[4], tiles[x[1]]) - x[3] if x[1] >= 0 else 0
        return 1700 + (2 if x[1] >= 0 else 1) * 4700 + min(a, b) * 3180 + (max(a, b) - min(a, b)) * 2400

    def page_order(self):
        """Whether the list is dealt out request by request first."""
        all_cycles, item, kv = int(self.cycles.sum()), self.mean_steps * 128 * self.row_bytes, self.tokens * self.kv_heads * self.row_bytes
        return (len(self.items) > SMS and all_cycles >= 225000 * SMS and self.mean_steps >= 9 and all_cycles >= 2.5 * self.cycles.max() * SMS
                and item * kv >= 8.4e6 ** 2)

    def end(self):
        return max(int(self.cycles[m].sum()) for m in self.mine)

    def longest_first(self):
        load = [0] * SMS
        for c in sorted(self.cycles[self.real].tolist(), reverse=True):
            heapq.heappush(load, heapq.heappop(load) + c)
        return max(load)

    def check(self):
        """Every item once, holes last and none in the first round."""
        assert sorted(map(tuple, self.work[self.real])) == sorted(map(tuple, self.items))
        assert len(self.work) <= SMS or len(self.work) % SMS == 0
        for m in self.mine:
            there = self.real[m]
            assert there[0] and not (np.diff(there.astype(int)) > 0).any()


def _batch(rng, requests, units, lo, hi, tail, again, shape):
    reqs = [[wl.unit(rng.randint(lo, hi), (r, k), recompute=range(min(again, lo))) for k in range(units)] + [tail] for r in range(requests)]
    return wl.build_workload("deal", shape, reqs, np.random.default_rng(1))


def _shape(heads, group, dim=128):
    return wl.ModelShape(heads * group, heads, dim, 64, 500000.0)


@pytest.mark.parametrize("seed", range(4))
def test_lists_whose_pages_need_no_order_are_dealt_longest_first(view, seed):
    """Short lists, lists of short items and of few pages: no block is later than longest first leaves it."""
    rng = random.Random(seed)
    dealt = 0
    for _ in range(15):
        w = _batch(rng, rng.randint(2, 40), rng.randint(1, 8), 40, rng.choice([60, 200, 500]), rng.randint(20, 250), rng.choice([4, 32]),
                   _shape(rng.choice([2, 4, 8]), rng.choice([2, 4, 5, 7, 8]), rng.choice([64, 128])))
        d = Deal(view, w)
        d.check()
        if len(d.items) > SMS and not d.page_order():
            assert d.end() == d.longest_first()
            dealt += 1
    assert dealt >= 5


@pytest.mark.parametrize("requests,units,again", [(4, 64, 32), (16, 16, 32), (32, 8, 160)])
def test_long_lists_over_many_pages_keep_to_few_requests_at_a_time(view, requests, units, again):
    """Over the first half of the rounds, the thread blocks' n-th items belong to three quarters of the requests at most."""
    d = Deal(view, _batch(random.Random(0), requests, units, 512, 512, 128, again, _shape(8, 4)))
    d.check()
    assert d.page_order() and d.end() <= 1.02 * d.longest_first()
    begin = d.work[:, 9]                       # first block-table entry: names the request
    for k in range(len(d.work) // SMS // 2):
        assert len(set(begin[[m[k] for m in d.mine]])) <= 3 * requests // 4


@pytest.mark.parametrize("requests,tail", [(1, 40), (6, 200), (20, 250)])
@pytest.mark.parametrize("blocks", [0, 1, 37, SMS - 16, SMS - 1, SMS, 2 * SMS])
def test_every_grid_a_launch_may_have_reaches_every_item(view, requests, tail, blocks):
    """Over the whole list and over every chunk: a block walks until its first hole, and what that leaves out is refused."""
    plan = tb.Plan(_batch(random.Random(requests), requests, 3, 100, 300, tail, 16, _shape(8, 4)), host_only=True)
    lists = {-1: np.zeros((view.view_work(plan._h, 0, None, 0), 12), np.int32)}
    view.view_work(plan._h, 0, lists[-1].ctypes.data, len(lists[-1]))
    grids = {c: view.view_grid(plan._h, c, blocks) for c in range(-1, view.view_chunks(plan._h))}
    plan.destroy()
    assert all(g > 0 for c, g in grids.items() if c >= 0)
    work, g = lists[-1], grids[-1]
    if g == 0:
        assert 0 < blocks < SMS < len(work)
        return
    reached = 0
    for b in range(g):
        for k in range(-(-len(work) // g)):
            i = k * g + (g - 1 - b if k & 1 else b)
            if i >= len(work):
                continue
            if work[i, 0] < 0:
                break
            reached += 1
    assert reached == (work[:, 0] >= 0).sum()
