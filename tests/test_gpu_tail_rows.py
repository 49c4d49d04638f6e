"""The last step of a request: value rows past its end, whatever the page held before, count for nothing."""
import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu
SCALE8 = 1 / 32


@pytest.mark.parametrize("dim,keys", [(64, "bf16"), (128, "bf16"), (128, "e4m3")])
@pytest.mark.parametrize("page", [32, 64, 128])
@pytest.mark.parametrize("tokens", [257, 263, 264, 287, 321, 383])     # page 128: 127, 121, 120, 97, 63 and 1 rows, odd ones among them
def test_rows_past_the_end_count_for_nothing(dim, keys, page, tokens):
    shape = wl.ModelShape(8, 2, dim, page, 10000.0)
    w = wl.build_workload("tail", shape, [[wl.unit(tokens - 9, "u", recompute=())] + [9], [wl.unit(100, "s", recompute=(0,))] + [tokens - 100]],
                          np.random.default_rng(tokens))
    plan = tb.Plan(w)
    t = wl.make_tensors(w, device="cuda:0", seed=6)
    page_off, pages, _ = plan.block_table()
    last = [int(pages[page_off[r + 1] - 1]) for r in range(w.batch)]
    outs = []
    for fill in (0.0, float("nan")):
        k, v = t.k_pool.clone(), t.v_pool.clone()
        plan.kv_compose(k, v)
        for r, p in enumerate(last):                   # the rows of the last page behind the request's end
            k[p, int(w.seq_len[r]) % page:], v[p, int(w.seq_len[r]) % page:] = fill, fill
        assert torch.isnan(v).any() == (fill != 0)
        out, lse = torch.zeros_like(t.q), torch.zeros(w.n_q, 8, device="cuda:0")
        if keys == "e4m3":
            k8 = (k.float() / SCALE8).to(torch.float8_e4m3fn).view(torch.uint8)
            plan.partial_prefill_attn_k8(k8, SCALE8, v, t.q, SCALE8, t.k_new, t.v_new, out, lse)
        else:
            plan.partial_prefill_attn(k, v, t.q, t.k_new, t.v_new, out, lse)
        outs.append((out, lse))
    assert plan.status() == 0
    assert torch.isfinite(outs[1][0]).all() and torch.isfinite(outs[1][1]).all()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    plan.destroy()
