"""The last step of a request: value rows past its end, whatever the page held before, count for nothing."""
import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("tokens", [257, 263, 264, 287, 320, 383, 384])     # 1 .. 127 rows and a whole step, odd ones among them
def test_rows_past_the_end_count_for_nothing(dim, tokens):
    shape = wl.ModelShape(8, 2, dim, 32, 10000.0)
    w = wl.build_workload("tail", shape, [[wl.unit(tokens - 9, "u", recompute=())] + [9], [wl.unit(100, "s", recompute=(0,))] + [tokens - 100]],
                          np.random.default_rng(tokens))
    plan = tb.Plan(w)
    t = wl.make_tensors(w, device="cuda:0", seed=6)
    outs = []
    for fill in (0.0, float("nan")):
        k, v = t.k_pool.clone(), t.v_pool.clone()
        page_off, pages, _ = plan.block_table()
        for r in range(w.batch):                       # the rows of the last page behind the request's end
            T, last = int(w.seq_len[r]), int(pages[page_off[r + 1] - 1])
            if T % 32:
                k[last, T % 32:], v[last, T % 32:] = fill, fill
        out, lse = torch.zeros_like(t.q), torch.zeros(w.n_q, 8, device="cuda:0")
        plan.kv_compose(k, v)
        plan.partial_prefill_attn(k, v, t.q, t.k_new, t.v_new, out, lse)
        outs.append((out, lse))
    assert plan.status() == 0
    assert torch.isfinite(outs[1][0]).all() and torch.isfinite(outs[1][1]).all()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    plan.destroy()
