"""What the composed-prefill library is timed on: the calls a serving program makes, over the range of
batches it makes them for.

A case describes a batch of prompts by plain numbers.  Every prompt is `head` tokens of its own, then
`units` context units of `unit_min` .. `unit_max` tokens, then `tail` tokens of its own; the prompt's own
tokens are always recomputed.  Of a cached unit either its first `prefix` tokens are recomputed or, with
`share` > 0, that share of its tokens at scattered offsets; a unit that missed (`miss` is the
probability) is recomputed whole.  `pool` > 0 draws the units from a pool of that many by Zipf popularity
(exponent `zipf`), so that requests share them; otherwise every unit is its own.  `stride` 1: keys were
cached rotated, 0: before rotation.  `layout` seeds lengths, popularity and offsets, which belong to the
case; page numbers and tensor contents come from the seed given to prepare().

`op` names the calls of one pass:
  layer      kv_compose + partial_prefill_attn: one layer of a batch, its plan made before
  extend     kv_compose + extend_write (missed units captured for the cache) + partial_prefill_attn
  prefill    Plan, `layers` layers, status and destroy: a whole batch from its descriptor on
  fp8_hit    kv_compose_from_fp8 + partial_prefill_attn: units kept as 8-bit floats
  fp8_store  kv_retain_fp8: the units of finished prompts go to the 8-bit store, position-free
  key8       kv_compose_k8 + partial_prefill_attn_k8: attention over 8-bit keys
  host       composed_prefill_host: activations in pinned host memory, both ways
  host_tier  composed_prefill_host_tier: cached units in a pinned host pool
"""
import math

import numpy as np
import torch

from paper_2609_32999_b200 import binding as tb
from paper_2609_32999_b200 import workloads as wl

DEVICE = "cuda"
SCALE8 = 1.0 / 32          # one e4m3 step of N(0, 1) data: codes reach 448 at 14 standard deviations

# (query heads, KV heads, head_dim, page size)
SHAPE_8B = dict(q_heads=32, kv_heads=8, head_dim=128, page=64, pairing=0, theta=500000.0)
SHAPE_70B = dict(q_heads=64, kv_heads=8, head_dim=128, page=64, pairing=0, theta=500000.0)
SHAPE_GROUP5 = dict(q_heads=40, kv_heads=8, head_dim=128, page=16, pairing=0, theta=1000000.0)
SHAPE_TINY = dict(q_heads=4, kv_heads=2, head_dim=64, page=16, pairing=0, theta=10000.0)


def _batch(requests, units, unit_min, unit_max, head, tail, prefix=0, share=0.0, miss=0.0, pool=0, zipf=1.0, stride=1, layers=1, layout=1):
    return dict(requests=requests, units=units, unit_min=unit_min, unit_max=unit_max, head=head, tail=tail, prefix=prefix,
                share=share, miss=miss, pool=pool, zipf=zipf, stride=stride, layers=layers, layout=layout)


def listed():
    return [
        # the smallest call: a short prompt of four snippets on a small model, all latency
        dict(name="tiny-layer", op="layer", **SHAPE_TINY, **_batch(1, 4, 64, 64, 16, 32, prefix=4)),
        # one question over ten retrieved passages, served alone: one layer of an 8B model
        dict(name="rag-one-layer", op="layer", **SHAPE_8B, **_batch(1, 10, 512, 512, 64, 128, prefix=16, pool=1000)),
        # sixteen agent turns, twenty memory records of odd lengths each, many of them shared
        dict(name="agent-memory-layer", op="layer", **SHAPE_8B, **_batch(16, 20, 128, 384, 256, 96, prefix=8, pool=5000, zipf=1.1)),
        # long-context retrieval: four prompts of 33 thousand tokens
        dict(name="long-rag-layer", op="layer", **SHAPE_8B, **_batch(4, 64, 512, 512, 0, 256, prefix=32, pool=4000, zipf=0.9)),
        # group of five heads, 16-token pages, keys cached before rotation, nothing aligned to anything
        dict(name="ragged-layer", op="layer", **SHAPE_GROUP5, **_batch(3, 7, 97, 911, 13, 77, prefix=5, stride=0)),
        # the largest call: a 70B model's mixed batch, a fifth of the units missed and captured for the cache
        dict(name="mixed-70b-extend", op="extend", **SHAPE_70B, **_batch(32, 12, 256, 1024, 0, 128, share=0.15, miss=0.2)),
        # time to first token of a lone question: the plan and all 32 layers
        dict(name="rag-one-prefill", op="prefill", **SHAPE_8B, **_batch(1, 10, 512, 512, 64, 128, prefix=16, pool=1000, layers=32)),
        # two long prompts whose units come from the 8-bit store
        dict(name="long-rag-fp8-hit", op="fp8_hit", **SHAPE_8B, **_batch(2, 64, 512, 512, 0, 256, prefix=32, pool=4000, zipf=0.9)),
        # the records of sixteen finished prompts go into the 8-bit store
        dict(name="agent-memory-fp8-store", op="fp8_store", **SHAPE_8B, **_batch(16, 20, 128, 384, 256, 96)),
        # two long prompts attended over 8-bit keys
        dict(name="long-rag-key8", op="key8", **SHAPE_8B, **_batch(2, 64, 512, 512, 0, 256, prefix=32, pool=4000, zipf=0.9)),
        # an engine whose activations live in host memory
        dict(name="long-rag-host", op="host", **SHAPE_8B, **_batch(4, 64, 512, 512, 0, 256, prefix=32, pool=4000, zipf=0.9)),
        # eight agent turns whose records sit in the node's host-memory cache
        dict(name="agent-memory-host-tier", op="host_tier", **SHAPE_8B, **_batch(8, 20, 128, 384, 256, 96, prefix=8, pool=5000, zipf=1.1)),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


_OPS = ["layer"] * 6 + ["extend"] * 2 + ["prefill"] * 2 + ["fp8_hit", "fp8_store", "key8", "host", "host_tier"]
_MOST_PAIR_FLOPS, _MOST_BYTES, _MOST_LINK_BYTES = 8e12, 2.5e9, 1.5e8


def draw(rng):
    """A case of the same ranges: any of the calls, 1 to 32 requests, 1 to 64 units of 32 to 1024 tokens, the
    model shapes the library takes."""
    while True:
        op = rng.choice(_OPS)
        dim = 128 if op == "key8" else rng.choice([64, 128, 128, 128])
        kv = rng.choice([2, 4, 8, 8])
        lo = _log_int(rng, 32, 640)
        case = dict(op=op, q_heads=kv * rng.choice([2, 4, 4, 5, 7, 8]), kv_heads=kv, head_dim=dim, page=rng.choice([16, 32, 64, 64]),
                    pairing=rng.choice([0, 0, 0, 1]), theta=rng.choice([10000.0, 500000.0, 1000000.0]),
                    **_batch(_log_int(rng, 1, 32), _log_int(rng, 1, 64), lo, rng.choice([lo, rng.randint(lo, min(1024, 4 * lo))]),
                             rng.choice([0, rng.randint(1, 256)]), _log_int(rng, 16, 256),
                             prefix=rng.randint(1, min(32, lo)), layers=rng.choice([16, 32, 48]) if op == "prefill" else 1,
                             layout=rng.randint(1, 1 << 20)))
        if op != "fp8_store":
            case["stride"] = rng.choice([1, 1, 1, 0])
            case["pool"] = rng.choice([0, 0, 1000, 5000])
            if op == "extend" or rng.random() < 0.25:
                case["share"] = round(rng.uniform(0.05, 0.2), 3)
                case["miss"] = round(rng.uniform(0.1, 0.3), 3)
        w = work(case)
        if w["flops"] > _MOST_PAIR_FLOPS or w["bytes"] > _MOST_BYTES or w["bytes"] < 2e5:
            continue
        if op in ("host", "host_tier") and w["bytes"] > _MOST_LINK_BYTES:
            continue
        return case


# ---- the batch a case describes

def _shape(case):
    return wl.ModelShape(case["q_heads"], case["kv_heads"], case["head_dim"], case["page"], case["theta"], rope_pairing=case["pairing"])


def _segments(case):
    """Per request, its segments in prompt order: lengths, popularity and offsets, all from the case."""
    rng = np.random.default_rng(case["layout"])
    lo, hi = case["unit_min"], case["unit_max"]
    pool_len = rng.integers(lo, hi + 1, size=case["pool"]) if case["pool"] else None
    fresh_id = 0
    requests = []
    for _ in range(case["requests"]):
        if case["pool"]:
            ids = wl.zipf_ranks(rng, case["units"], case["pool"], case["zipf"], distinct=True)
            named = [(("p", k), int(pool_len[k - 1])) for k in ids]
        else:
            named = [(("u", fresh_id + k), int(n)) for k, n in enumerate(rng.integers(lo, hi + 1, size=case["units"]))]
            fresh_id += case["units"]
        segs = [case["head"]] if case["head"] else []
        for uid, n in named:
            cached = bool(rng.random() >= case["miss"])
            if case["share"]:
                again = np.sort(rng.choice(n, size=max(1, int(round(case["share"] * n))), replace=False))
            else:
                again = range(min(case["prefix"], n))
            segs.append(wl.unit(n, uid, cached=cached, stride=case["stride"], recompute=again))
        segs.append(case["tail"])
        requests.append(segs)
    return requests


def _workload(case, seed):
    """The descriptor of the batch: layout from the case, page numbers from the seed."""
    w = wl.build_workload(case["op"], _shape(case), _segments(case), np.random.default_rng(seed))
    if case["op"] in ("fp8_hit", "key8", "host_tier"):
        # the units live in a pool of their own: number its pages from 0
        used, w.unit_pages = np.unique(w.unit_pages, return_inverse=True)
        w.unit_pages = w.unit_pages.astype(np.int32)
        w.num_source_pages = max(1, len(used))
    if case["op"] == "extend":
        _capture_missed_units(w)
    return w


def _capture_missed_units(w):
    """Marks every missed unit for the cache; its pages are appended to the pool."""
    off, pages, page = [0], [], w.num_pool_pages
    for u in range(len(w.unit_len)):
        if w.unit_page_off[u + 1] == w.unit_page_off[u]:
            n = -(-int(w.unit_len[u]) // w.shape.page_size)
            pages.extend(range(page, page + n))
            page += n
        off.append(len(pages))
    w.unit_retain_page_off, w.unit_retain_pages = np.array(off, np.int32), np.array(pages, np.int32)
    w.num_pool_pages = page


def _store_workload(case, seed):
    """Cache entries read out of finished prompts: entry = one unit, found in the middle of its prompt's pages,
    written without rotation."""
    rng = np.random.default_rng(seed)
    B = case["page"]
    prompts = _segments(case)
    lengths = [sum(s if isinstance(s, int) else s.length for s in segs) for segs in prompts]
    n_src = sum(-(-t // B) for t in lengths)
    src_perm = rng.permutation(n_src)
    u_len, u_pos, u_off, page_off, pages = [], [], [], [0], []
    first = 0
    for segs, t in zip(prompts, lengths):
        p = 0
        for s in segs:
            n = s if isinstance(s, int) else s.length
            if not isinstance(s, int):
                u_len.append(n); u_pos.append(p); u_off.append(p % B)
                pages.extend(int(src_perm[first + k]) for k in range(p // B, (p + n - 1) // B + 1))
                page_off.append(len(pages))
            p += n
        first += -(-t // B)
    n_dst = sum(-(-n // B) for n in u_len)
    i32 = lambda x: np.ascontiguousarray(np.asarray(x, dtype=np.int32))   # noqa: E731
    k = len(u_len)
    return wl.Workload(name="store", shape=_shape(case), seq_len=i32(u_len), unit_off=i32(range(k + 1)), unit_len=i32(u_len),
                       unit_cached_pos=i32(u_pos), unit_cached_stride=i32([1] * k), unit_target_pos=i32([0] * k),
                       unit_page_off=i32(page_off), unit_pages=i32(pages), recompute_off=i32([0] * (k + 1)), recompute_pos=i32([]),
                       free_pages=i32(rng.permutation(n_dst)), num_pool_pages=n_dst, unit_src_offset=i32(u_off),
                       unit_target_stride=i32([0] * k), num_source_pages=n_src)


def work(case):
    """Bytes: every distinct cached row read once, every assembled row written once, fresh rows, queries, outputs and
    log-sums once each.  Flops: 4 x head_dim per unmasked (query, key) pair and query head."""
    kv_row = 2 * case["kv_heads"] * case["head_dim"]            # K and V elements of one token
    if case["op"] == "fp8_store":
        tokens = sum(s.length for segs in _segments(case) for s in segs if not isinstance(s, int))
        return {"bytes": tokens * kv_row * 3, "flops": 0}
    distinct, cached, n_q, pairs, captured = {}, 0, 0, 0, 0
    for segs in _segments(case):
        p = 0
        for s in segs:
            if isinstance(s, int):
                offs, n = np.arange(s), s
            elif s.cached:
                offs, n = np.asarray(list(s.recompute), dtype=np.int64), s.length
                distinct[s.uid] = n
                cached += n
            else:
                offs, n = np.arange(s.length), s.length
                captured += n
            n_q += len(offs)
            pairs += int((p + offs + 1).sum())
            p += n
    q_row = case["q_heads"] * case["head_dim"]
    src_bytes = 1 if case["op"] == "fp8_hit" else 2
    key_bytes = 1 if case["op"] == "key8" else 2
    total = sum(distinct.values()) * kv_row * src_bytes + (cached + n_q) * kv_row * (2 + key_bytes) // 2 + n_q * kv_row * 2
    total += n_q * (q_row * 4 + case["q_heads"] * 4)
    if case["op"] == "extend":
        total += captured * kv_row * 2 + n_q * q_row * 2        # captured rows written, rotated queries written
    return {"bytes": total * case["layers"], "flops": 4 * q_row * pairs * case["layers"]}


def tolerance(case):
    """Four times what attention outputs differ by from fp64 attention over the same pages: 7e-4 .. 2e-3 in the 2-norm,
    1e-2 .. 2.6e-2 at most (keys, probabilities and outputs are rounded to bf16).  8-bit codes of rotated keys flip at
    ties, fewer than one in a thousand; the codes of values are exact."""
    if case["op"] in ("fp8_store", "key8"):
        return {"rel": 8e-3, "max": 0.1, "differ": 2e-3}
    return {"rel": 8e-3, "max": 0.1}


# ---- what a program holds before the call, and the call

def _bf16(gen, *dims):
    out = torch.empty(*dims, dtype=torch.bfloat16, device=DEVICE)
    return out.normal_(generator=gen)


def _codes(gen, *dims):
    """N(0, 1) values as e4m3 codes of step SCALE8."""
    return (_bf16(gen, *dims).float() * (1.0 / SCALE8)).to(torch.float8_e4m3fn).view(torch.uint8)


class State:
    """Tensors, descriptor and plan of one batch."""


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    op = case["op"]
    s = State()
    s.op, s.layers = op, case["layers"]
    s.w = w = _store_workload(case, seed) if op == "fp8_store" else _workload(case, seed)
    B, Hkv, Hq, D = case["page"], case["kv_heads"], case["q_heads"], case["head_dim"]
    dst, src = (w.num_pool_pages, B, Hkv, D), (w.num_source_pages, B, Hkv, D)
    if op == "fp8_store":
        s.k_src, s.v_src = _bf16(gen, *src), _bf16(gen, *src)
        s.k8, s.v8 = (torch.zeros(dst, dtype=torch.uint8, device=DEVICE) for _ in range(2))
        s.plan = tb.Plan(w)
        return s
    n_q, L = w.n_q, case["layers"]
    if op == "prefill":
        s.k, s.v = _bf16(gen, L, *dst), _bf16(gen, L, *dst)
        s.q, s.k_new, s.v_new = _bf16(gen, L, n_q, Hq, D), _bf16(gen, L, n_q, Hkv, D), _bf16(gen, L, n_q, Hkv, D)
        s.out = torch.empty(L, n_q, Hq, D, dtype=torch.bfloat16, device=DEVICE)
        s.lse = torch.empty(L, n_q, Hq, dtype=torch.float32, device=DEVICE)
        return s
    s.v = _bf16(gen, *dst)
    s.k = torch.zeros(dst, dtype=torch.uint8, device=DEVICE) if op == "key8" else _bf16(gen, *dst)
    s.q, s.k_new, s.v_new = _bf16(gen, n_q, Hq, D), _bf16(gen, n_q, Hkv, D), _bf16(gen, n_q, Hkv, D)
    s.out = torch.empty(n_q, Hq, D, dtype=torch.bfloat16, device=DEVICE)
    s.lse = torch.empty(n_q, Hq, dtype=torch.float32, device=DEVICE)
    if op == "fp8_hit":
        s.k_src, s.v_src = _codes(gen, *src), _codes(gen, *src)
    elif op == "key8":
        s.k_src, s.v_src = _bf16(gen, *src), _bf16(gen, *src)
    elif op == "host_tier":
        s.k_src, s.v_src = _bf16(gen, *src).cpu().pin_memory(), _bf16(gen, *src).cpu().pin_memory()
    elif op == "host":
        s.q, s.k_new, s.v_new, s.out, s.lse = (t.cpu().pin_memory() for t in (s.q, s.k_new, s.v_new, s.out, s.lse))
    s.plan = tb.Plan(w)
    return s


def run(s):
    if s.op == "layer":
        s.plan.kv_compose(s.k, s.v)
        s.plan.partial_prefill_attn(s.k, s.v, s.q, s.k_new, s.v_new, s.out, s.lse)
    elif s.op == "extend":
        # the projections arrive un-rotated; q is rotated in place
        s.plan.kv_compose(s.k, s.v)
        s.plan.extend_write(s.k, s.v, s.q, s.k_new, s.v_new, s.k, s.v)
        s.plan.partial_prefill_attn(s.k, s.v, s.q, None, None, s.out, s.lse)
    elif s.op == "prefill":
        plan = tb.Plan(s.w)
        for l in range(s.layers):
            plan.kv_compose(s.k[l], s.v[l])
            plan.partial_prefill_attn(s.k[l], s.v[l], s.q[l], s.k_new[l], s.v_new[l], s.out[l], s.lse[l])
        status = plan.status()           # waits for the batch, as a server does before it samples the first token
        plan.destroy()
        return {"k": s.k, "v": s.v, "out": s.out, "lse": s.lse, "status": status}
    elif s.op == "fp8_hit":
        s.plan.kv_compose_from_fp8(s.k_src, s.v_src, SCALE8, SCALE8, s.k, s.v)
        s.plan.partial_prefill_attn(s.k, s.v, s.q, s.k_new, s.v_new, s.out, s.lse)
    elif s.op == "fp8_store":
        s.plan.kv_retain_fp8(s.k_src, s.v_src, s.k8, s.v8, SCALE8, SCALE8)
        return {"k8": s.k8, "v8": s.v8}
    elif s.op == "key8":
        s.plan.kv_compose_k8(s.k_src, s.v_src, s.k, s.v, SCALE8)
        s.plan.partial_prefill_attn_k8(s.k, SCALE8, s.v, s.q, SCALE8, s.k_new, s.v_new, s.out, s.lse)
    elif s.op == "host":
        s.plan.composed_prefill_host(s.k, s.v, s.q, s.k_new, s.v_new, s.out, s.lse)
    elif s.op == "host_tier":
        s.plan.composed_prefill_host_tier(s.k_src, s.v_src, s.k, s.v, s.q, s.k_new, s.v_new, s.out, s.lse)
    else:
        raise ValueError(s.op)
    result = {"k": s.k, "v": s.v, "out": s.out, "lse": s.lse}
    if s.op == "extend":
        result["q"] = s.q
    return result


# ---- the same outputs in 64 bits

def _rotated(x, pos, case):
    """Rows x [n, heads, D] turned by pos [n] positions."""
    D = case["head_dim"]
    freq = case["theta"] ** (-2.0 * torch.arange(D // 2, dtype=torch.float64, device=DEVICE) / D)
    ang = pos.double()[:, None, None] * freq
    c, n = ang.cos(), ang.sin()
    lo, hi = (x[..., 0::2], x[..., 1::2]) if case["pairing"] else (x[..., :D // 2], x[..., D // 2:])
    a, b = lo * c - hi * n, hi * c + lo * n
    return torch.stack((a, b), dim=-1).flatten(-2) if case["pairing"] else torch.cat((a, b), dim=-1)


def _attended(q, k, v, pos, scale):
    """Rows q [n, Hq, D] at positions pos over keys and values [T, Hkv, D]: outputs and log-sums."""
    n, Hq, D = q.shape
    T, Hkv = k.shape[:2]
    g = Hq // Hkv
    out, lse = torch.empty_like(q), q.new_empty(n, Hq)
    rows = max(1, (1 << 28) // (T * g))
    at = torch.arange(T, device=q.device)
    for h in range(Hkv):
        for r in range(0, n, rows):
            x = q[r:r + rows, h * g:(h + 1) * g]
            score = (x.reshape(-1, D) @ k[:, h].T).view(-1, g, T) * scale
            score.masked_fill_(at > pos[r:r + rows, None, None], -math.inf)
            total = score.logsumexp(-1)
            lse[r:r + rows, h * g:(h + 1) * g] = total
            out[r:r + rows, h * g:(h + 1) * g] = (score.sub_(total[..., None]).exp_().view(-1, T) @ v[:, h]).view(-1, g, D)
    return out, lse


def exact(case, seed):
    """The outputs of run() in fp64, nothing rounded on the way; None for 8-bit codes."""
    op, B = case["op"], case["page"]
    if op == "fp8_store":
        return None
    s = prepare(case, seed)
    w = s.w
    gpu = lambda x: torch.as_tensor(np.asarray(x), dtype=torch.int64, device=DEVICE)   # noqa: E731
    T = w.seq_len
    page_off = np.concatenate([[0], np.cumsum(-(-T // B))])
    slots = [gpu(w.free_pages[page_off[r] + np.arange(T[r]) // B].astype(np.int64) * B + np.arange(T[r]) % B) for r in range(len(T))]
    pos = [gpu(w.recompute_pos[w.recompute_off[r]:w.recompute_off[r + 1]]) for r in range(len(T))]
    src, dst, shift, kept, kept_row = [], [], [], [], []
    for r in range(len(T)):
        for u in range(w.unit_off[r], w.unit_off[r + 1]):
            i, first = np.arange(w.unit_len[u]), w.unit_page_off[u]
            if w.unit_page_off[u + 1] > first:
                src.append(gpu(w.unit_pages[first + i // B].astype(np.int64) * B + i % B))
                dst.append(slots[r][w.unit_target_pos[u]:w.unit_target_pos[u] + len(i)])
                shift.append(gpu(w.unit_target_pos[u] + i - w.unit_cached_pos[u] - w.unit_cached_stride[u] * i))
            elif op == "extend":
                pages = w.unit_retain_pages[w.unit_retain_page_off[u]:]
                kept.append(gpu(pages[i // B].astype(np.int64) * B + i % B))
                row = w.recompute_off[r] + np.searchsorted(w.recompute_pos[w.recompute_off[r]:w.recompute_off[r + 1]], w.unit_target_pos[u])
                kept_row.append(gpu(row + i))
    fresh = torch.cat([slots[r][pos[r]] for r in range(len(T))])

    def layer(k, v, k_src, v_src, q, k_new, v_new):
        rows = lambda t: t.to(DEVICE).flatten(0, 1).double()                           # noqa: E731
        D = case["head_dim"]
        k, v, q, k_raw, v_new = rows(k), rows(v), q.to(DEVICE).double(), k_new.to(DEVICE).double(), v_new.to(DEVICE).double()
        if src:
            at, to = torch.cat(src), torch.cat(dst)
            if k_src is None:
                rk, rv = k[at], v[at]
            else:
                rk, rv = ((t.to(DEVICE).flatten(0, 1)[at].view(torch.float8_e4m3fn).double() * SCALE8) if t.dtype == torch.uint8 else
                          t.to(DEVICE).flatten(0, 1)[at].double() for t in (k_src, v_src))
            k[to], v[to] = _rotated(rk, torch.cat(shift), case), rv
        k_new = k_raw
        if op == "extend":
            every = torch.cat(pos)
            q, k_new = _rotated(q, every, case), _rotated(k_raw, every, case)
        k[fresh], v[fresh] = k_new, v_new
        if kept:
            k[torch.cat(kept)], v[torch.cat(kept)] = k_raw[torch.cat(kept_row)], v_new[torch.cat(kept_row)]
        parts = [_attended(q[w.recompute_off[r]:w.recompute_off[r + 1]], k[slots[r]], v[slots[r]], pos[r], 1.0 / math.sqrt(D))
                 for r in range(len(T))]
        pool = (-1, B) + tuple(k.shape[1:])
        return k.view(pool), v.view(pool), torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]), q

    k_src, v_src = getattr(s, "k_src", None), getattr(s, "v_src", None)
    if op == "prefill":
        each = [layer(s.k[l], s.v[l], None, None, s.q[l], s.k_new[l], s.v_new[l]) for l in range(s.layers)]
        k, v, out, lse, _ = (torch.stack(t) for t in zip(*each))
        return {"k": k, "v": v, "out": out, "lse": lse, "status": None}
    k, v, out, lse, q = layer(s.k, s.v, k_src, v_src, s.q, s.k_new, s.v_new)
    result = {"k": None if op == "key8" else k, "v": v, "out": out, "lse": lse}
    if op == "extend":
        result["q"] = q
    return result
