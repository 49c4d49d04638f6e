"""The rule that cuts key ranges (split-KV) over batches of every size, against a plain restatement of it: the planner
prunes and shortens the search, and must find the same cut."""
import heapq
import random

import numpy as np
import pytest

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

SMS, MIN_STEPS, MAX_PARTS, ROUNDS = 148, 2, 32, 4


def _cycles(a, b, tiles):
    both = min(a, b)
    return 1700 + tiles * 4700 + both * 3180 + (max(a, b) - both) * 2400


def _pairs(w):
    """(steps of the first tile or None, steps of the longer one) of every tile pair."""
    tok = 128 // (w.shape.num_q_heads // w.shape.num_kv_heads)
    pairs = []
    for r in range(len(w.seq_len)):
        pos = w.recompute_pos[w.recompute_off[r]:w.recompute_off[r + 1]]
        steps = [(int(pos[min(j + tok, len(pos)) - 1]) + 1 + 127) // 128 for j in range(0, len(pos), tok)]
        pairs += [(steps[k], steps[k + 1]) if k + 1 < len(steps) else (None, steps[k]) for k in range(0, len(steps), 2)]
    return pairs


def _parts(steps, limit):
    return max(1, min(-(-steps // limit), MAX_PARTS, steps // MIN_STEPS))


def _lengths(steps, limit):
    parts = _parts(steps, limit)
    n = -(-steps // parts)
    return [(b, min(steps, b + n)) for b in range(0, steps, n)]


def _modelled(pairs, heads, limit):
    cost, slots = [], 0
    for a, b in pairs:
        cuts = _lengths(b, limit)
        for lo, hi in cuts:
            n_a = max(0, min(a or 0, hi) - lo)
            cost += [_cycles(n_a, hi - lo, 2 if n_a else 1)] * heads
            slots += (2 if n_a else 1) * heads if _parts(b, limit) > 1 else 0
    load = [0] * SMS
    for c in sorted(cost, reverse=True):
        heapq.heappush(load, heapq.heappop(load) + c)
    return max(load) + ((4500 if len(cost) <= SMS else 9000) + slots * 20 if slots else 0)


def _limit(pairs, heads):
    """Most steps a part may have; the longest tile's where nothing is cut."""
    count = lambda limit: heads * sum(_parts(b, limit) for _, b in pairs)          # noqa: E731
    longest = max([b for _, b in pairs], default=1)
    limit, uncut = longest, len(pairs) * heads
    if 0 < 2 * uncut <= SMS:
        low = longest
        while low > MIN_STEPS and count(low - 1) <= SMS:
            low -= 1
        if _modelled(pairs, heads, low) < _modelled(pairs, heads, longest) * 90 // 100:
            limit = low
    elif 0 < uncut <= ROUNDS * SMS:
        best = _modelled(pairs, heads, longest) * 90 // 100
        low = longest * 3 // 4
        while low >= 2 * MIN_STEPS and count(low) <= 2 * ROUNDS * SMS:
            m = _modelled(pairs, heads, low)
            if m < best:
                best, limit = m, low
            low = low * 5 // 6
    return limit


def items_and_cut(w):
    pairs, heads = _pairs(w), w.shape.num_kv_heads
    limit = _limit(pairs, heads)
    return heads * sum(len(_lengths(b, limit)) for _, b in pairs), limit < max([b for _, b in pairs], default=1)


def is_chained(w):
    """Whether the plan's kernels are launched with programmatic serialization: its attention is modelled short."""
    pairs, heads = _pairs(w), w.shape.num_kv_heads
    limit, total = _limit(pairs, heads), 0
    for a, b in pairs:
        for lo, hi in _lengths(b, limit):
            n_a = max(0, min(a or 0, hi) - lo)
            total += _cycles(n_a, hi - lo, 2 if n_a else 1) * heads
    return total // SMS <= 300000


@pytest.mark.parametrize("seed", range(6))
def test_the_planner_cuts_as_the_rule_says(seed):
    rng = random.Random(seed)
    cut = 0
    for i in range(20):
        heads, group = rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 4, 5, 8])
        shape = wl.ModelShape(heads * group, heads, rng.choice([64, 128]), 64, 500000.0)
        units = max(1, int(2 ** rng.uniform(0, 6)))
        reqs = [[wl.unit(rng.choice([128, 500, 512]), (r, k), recompute=range(rng.choice([0, 4]))) for k in range(units)] + [rng.randint(1, 200)]
                for r in range(max(1, int(2 ** rng.uniform(0, 4.6))))]
        w = wl.build_workload("cut", shape, reqs, np.random.default_rng(i))
        plan = tb.Plan(w, host_only=True)
        want, was_cut = items_and_cut(w)
        assert plan.info.n_attn_items == want, (i, len(reqs), units, heads, group)
        cut += was_cut
    assert 3 <= cut <= 17                  # both sides of the rule
