"""The attention work list over batch sizes at which its rules change: a lone tile cut into more parts than one
batch of the merge holds, lists that fit the SMs once, lists of one to four rounds (cut when that is modelled
faster), lists left alone."""
import numpy as np
import pytest

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SHAPE_128 = wl.ModelShape(32, 8, 128, 64, 500000.0)
SHAPE_64 = wl.ModelShape(10, 2, 64, 16, 10000.0)          # five heads per group: padding rows in every tile
SHAPE_1 = wl.ModelShape(4, 1, 128, 32, 500000.0)


@pytest.mark.parametrize("shape,requests,unit,units,tail,items", [
    (SHAPE_1, 1, 3000, 2, 9, (9, 148)),           # one tile of 47 steps: more parts than one batch of the merge
    (SHAPE_1, 1, 129, 1, 1, (1, 1)),              # too short to be cut
    (SHAPE_64, 1, 900, 5, 40, (5, 148)),
    (SHAPE_64, 7, 300, 3, 30, (15, 148)),
    (SHAPE_128, 5, 700, 3, 120, (81, 592)),       # 80 uncut items: more than half the SMs
    (SHAPE_128, 10, 500, 4, 70, (160, 592)),      # two rounds uncut
    (SHAPE_128, 1, 200, 2, 500, (64, 148)),       # a dense tail: hundreds of fresh rows in one item's key range
])
def test_parity_where_the_work_list_changes(shape, requests, unit, units, tail, items):
    rng = np.random.default_rng(3)
    reqs = [[3] + [wl.unit(unit + 7 * r, ("u", r, i), recompute=(0, 5, unit // 2)) for i in range(units)] + [tail + r] for r in range(requests)]
    w = wl.build_workload("split", shape, reqs, rng)
    n = tb.Plan(w, host_only=True).info.n_attn_items
    assert items[0] <= n <= items[1], n
    g = gu.run_layer(w, seed=31)
    assert g.status == 0
    asm, _, _ = gu.check_assembled(g)
    gu.check_untouched(g)
    gu.check_attention(g, asm)
