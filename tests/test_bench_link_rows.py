"""Bytes over the link in the bench's host-tier record: the reader fetches a unit that several requests use once."""
import numpy as np
import pytest

import bench
from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl


@pytest.mark.parametrize("make", [lambda: wl.config(2), lambda: wl.config(3, requests_override=6),
                                  lambda: wl.build_workload("shared", wl.ModelShape(8, 2, 64, 16, 10000.0),
                                                            [[3] + [wl.unit(40 + i, ("s", i), recompute=(0,)) for i in (0, r, 3)] + [9] for r in range(3)],
                                                            np.random.default_rng(2))])
def test_every_unit_counts_once(make):
    w = make()
    src = tb.Plan(w, host_only=True).block_table()[2]
    assert bench.distinct_cached_tokens(w) == len(np.unique(src[src >= 0])) <= w.cached_tokens
