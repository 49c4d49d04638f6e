"""Units used by several requests (and twice by one): the host-tier reader fetches their rows once and writes
them for every user.  Bits of the plain gather, for both pairings, head sizes and cached forms."""
import copy

import numpy as np
import pytest
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,pairing,page", [(128, 0, 64), (64, 1, 16), (128, 1, 32), (64, 0, 8)])
@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("requests", [1, 3, 9])
def test_rows_fetched_once_for_all_users(dim, pairing, page, fp8, requests):
    shape = wl.ModelShape(8, 2, dim, page, 10000.0, rope_pairing=pairing)
    rng = np.random.default_rng(dim + page + requests)
    n = [1, 33, 100, 31, 200]
    reqs = []
    for r in range(requests):
        ids = rng.permutation(5)[:4].tolist()
        ids.append(ids[0])                                     # one unit twice in a request
        segs = [int(rng.integers(1, 20))]
        # unit 3 appears cached before rotation, the others rotated
        segs += [wl.unit(n[i], ("s", i), stride=0 if i == 3 else 1, recompute=(0,)) for i in ids]
        reqs.append(segs + [int(rng.integers(1, 30))])
    w = wl.build_workload("shared", shape, reqs, rng)
    w = copy.copy(w)
    w.num_source_pages = w.num_pool_pages
    t = wl.make_tensors(w, device="cuda:0", seed=5)
    if fp8:
        src = [(x.float() * 32).to(torch.float8_e4m3fn).view(torch.uint8).cpu().pin_memory() for x in (t.k_pool, t.v_pool)]
        extra = dict(src_format=1, k_scale=1 / 32, v_scale=1 / 32)
    else:
        src, extra = [x.cpu().pin_memory() for x in (t.k_pool, t.v_pool)], {}
    plan = tb.Plan(w)
    pools = [[torch.zeros_like(t.k_pool), torch.zeros_like(t.v_pool)] for _ in range(2)]
    outs = [torch.zeros_like(t.q) for _ in range(2)]
    if fp8:
        plan.kv_compose_from_fp8(*src, 1 / 32, 1 / 32, *pools[0])
    else:
        plan.kv_compose_from(*src, *pools[0])
    plan.partial_prefill_attn(*pools[0], t.q, t.k_new, t.v_new, outs[0], None)
    plan.composed_prefill_host_tier(*src, *pools[1], t.q, t.k_new, t.v_new, outs[1], None, **extra)
    torch.cuda.synchronize()
    assert plan.status() == 0
    assert torch.equal(pools[0][0], pools[1][0]) and torch.equal(pools[0][1], pools[1][1])
    assert torch.equal(outs[0], outs[1])
