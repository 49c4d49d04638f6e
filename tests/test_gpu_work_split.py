"""The attention work list over batch sizes at which its rules change: a lone tile cut into more parts than one
batch of the merge holds, lists that fit the SMs once, lists of one to four rounds (cut when that is modelled
faster), lists left alone."""
import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl
from tests import gpu_util as gu
from tests.test_cut_rule import items_and_cut

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


@pytest.mark.parametrize("requests,units,tail,uncut,items", [
    (20, 6, 60, 160, 640),                        # one to two rounds, cut
    (38, 8, 20, 304, 912),                        # two to four rounds, cut
    (57, 8, 4, 456, 456),                         # three to four rounds, left alone
    (75, 3, 20, 600, 600),                        # more than four rounds: never cut
])
def test_parity_of_lists_of_several_rounds(requests, units, tail, uncut, items):
    shape = wl.ModelShape(8, 8, 64, 64, 500000.0)
    rng = np.random.default_rng(11)
    reqs = [[3] + [wl.unit(1024, (r % 4, i), recompute=()) for i in range(units)] + [tail] for r in range(requests)]
    w = wl.build_workload("rounds", shape, reqs, rng)
    assert items_and_cut(w) == (items, items > uncut) and tb.Plan(w, host_only=True).info.n_attn_items == items
    g = gu.run_layer(w, seed=7)
    assert g.status == 0
    checked = [0, requests // 2, requests - 1]
    asm, _, _ = gu.check_assembled(g, requests=checked)
    gu.check_attention(g, asm, {r: gu.sample_rows(w, r, rng, 0, 8) for r in checked})


@pytest.mark.parametrize("heads,kv_heads,dim,fresh", [
    (7, 1, 128, 1), (7, 1, 128, 2), (14, 2, 128, 5),      # 7, 14 and 35 rows: less than one group of 16, and a remainder
    (3, 1, 64, 11), (16, 1, 64, 8), (16, 2, 128, 17),     # 33 rows; a full tile; a full tile and one row
])
def test_merge_of_row_groups(heads, kv_heads, dim, fresh):
    """Cut lists whose tiles end inside a group of 16 rows, both head sizes."""
    shape = wl.ModelShape(heads, kv_heads, dim, 32, 10000.0)
    rng = np.random.default_rng(5)
    w = wl.build_workload("merge", shape, [[wl.unit(1500, ("u", i), recompute=()) for i in range(2)] + [fresh]], rng)
    assert items_and_cut(w)[1]
    g = gu.run_layer(w, seed=17)
    assert g.status == 0
    asm, _, _ = gu.check_assembled(g)
    gu.check_untouched(g)
    gu.check_attention(g, asm)


@pytest.mark.parametrize("masked_steps", [2, 9, 20])
def test_parts_whose_scores_all_overflow_count_for_nothing(masked_steps):
    """Scores of -inf in whole parts of a cut key range - more parts than the merge reads at once, too - leave the
    later parts their weight: with equal finite scores the output is the mean of the visible finite keys' values."""
    w = wl.build_workload("overflow", SHAPE_1, [[3] + [wl.unit(3000, ("u", i), recompute=(0, 5, 1500)) for i in range(2)] + [9]],
                          np.random.default_rng(3))
    plan = tb.Plan(w)
    assert plan.info.n_attn_items == 16                    # 47 steps in parts of three
    t = wl.make_tensors(w, device="cuda:0", seed=4)
    page_off, pages, _ = plan.block_table()
    T, B, dead = int(w.seq_len[0]), SHAPE_1.page_size, 128 * masked_steps
    at = torch.from_numpy(pages[np.arange(T) // B].astype(np.int64) * B + np.arange(T) % B).to("cuda:0")
    # q k = -1e40 a pair in the first `dead` keys, about 1 (the same everywhere) in the others
    t.q.fill_(1e20)
    k = t.k_pool.flatten(0, 1)
    k[at[:dead]], k[at[dead:]] = -1e20, 1e-20
    pos = torch.from_numpy(w.recompute_pos.astype(np.int64)).to("cuda:0")
    v = t.v_pool.flatten(0, 1)
    v[at] = torch.randn(T, *v.shape[1:], device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(1)).to(torch.bfloat16)
    out, lse = torch.zeros_like(t.q), torch.zeros(w.n_q, SHAPE_1.num_q_heads, device="cuda:0")
    plan.partial_prefill_attn(t.k_pool, t.v_pool, t.q, None, None, out, lse)
    assert plan.status() == 0
    score = 128 * float(t.q[0, 0, 0]) * float(k[at[dead], 0, 0]) / 128 ** 0.5
    seen = 0
    for j, p in enumerate(pos.tolist()):
        if p < dead:
            continue
        want = v[at[dead:p + 1]].double().mean(0)           # one KV head: the same for all query heads
        # probabilities are 2^x of one common x: each rounded to bf16 alike, outputs rounded once (2^-9)
        assert torch.allclose(out[j].double(), want.expand(SHAPE_1.num_q_heads, -1), rtol=2 ** -7, atol=1e-4), (j, p)
        assert torch.allclose(lse[j].double(), torch.full_like(lse[j].double(), score + np.log(p + 1 - dead)), rtol=1e-4), (j, p)
        seen += 1
    assert seen >= 9
    plan.destroy()
