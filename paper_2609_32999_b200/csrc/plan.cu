// Host-side placement: validation of a batch descriptor and construction of every table the
// kernels read (Sec. 5.3 "Placement before preparation"; storage blocks of Sec. 5.1).
// Pure host code: it makes no CUDA call, so it also runs where no GPU exists.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <functional>
#include <numeric>
#include <tuple>

#include <vector_types.h>

#include "plan.h"

namespace tessera {

namespace {

std::string fmt(const char *f, long a = 0, long b = 0, long c = 0) {
    char buf[256];
    snprintf(buf, sizeof buf, f, a, b, c);
    return buf;
}

// Merge of a split list in SM cycles: the launch and its first loads, and 65 KB of partial results per slot
// written and read back through L2.
constexpr int64_t kMergeCycles = 9000, kMergeCyclesOneRound = 4500, kMergeCyclesPerSlot = 20;

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

}  // namespace

int32_t build_plan_host(const tessera_model_cfg *cfg, const tessera_compose_desc *d,
                        int32_t num_pool_pages, int num_sms, bool may_cut, tessera_plan *pl, std::string *err) {
    auto fail = [&](int32_t code, const std::string &msg) { *err = msg; return code; };
    if (!cfg || !d || !pl) return fail(TESSERA_INVALID_ARG, "null cfg / desc / plan");
    if (num_sms <= 0) return fail(TESSERA_INVALID_ARG, "multiprocessor count must be positive");
    pl->num_sms = num_sms;
    if (d->batch < 0 || num_pool_pages < 0 || d->n_free < 0)
        return fail(TESSERA_INVALID_ARG, "negative batch, pool size or free-list length");
    if (d->batch > 0 && (!d->seq_len || !d->unit_off || !d->recompute_off))
        return fail(TESSERA_INVALID_ARG, "null seq_len / unit_off / recompute_off");

    // ---- shapes the kernels cover
    const int Hq = cfg->num_q_heads, Hkv = cfg->num_kv_heads, D = cfg->head_dim, B = cfg->page_size;
    if (Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0)
        return fail(TESSERA_UNSUPPORTED_SHAPE, fmt("num_q_heads %ld must be a positive multiple of num_kv_heads %ld", Hq, Hkv));
    if (Hq / Hkv > 16) return fail(TESSERA_UNSUPPORTED_SHAPE, "group size H_q/H_kv above 16");
    if (D != 64 && D != 128) return fail(TESSERA_UNSUPPORTED_SHAPE, fmt("head_dim %ld: only 64 and 128", D));
    if (B <= 0 || B % 8 != 0 || B > 128 || !is_pow2(B))
        return fail(TESSERA_UNSUPPORTED_SHAPE, fmt("page_size %ld: a power of two in 8..128", B));
    if (cfg->rope_pairing != 0 && cfg->rope_pairing != 1)
        return fail(TESSERA_UNSUPPORTED_SHAPE, "rope_pairing: 0 (half-split pairs) or 1 (interleaved pairs)");
    if (!cfg->inv_freq && !(cfg->rope_theta > 0.0)) return fail(TESSERA_INVALID_ARG, "rope_theta must be positive");
    if ((int64_t)num_pool_pages * B > (int64_t)INT32_MAX)
        return fail(TESSERA_UNSUPPORTED_SHAPE, "pool has more than 2^31 slots");

    pl->cfg = *cfg;
    pl->inv_freq.resize(D / 2);
    for (int m = 0; m < D / 2; ++m)
        pl->inv_freq[m] = cfg->inv_freq ? cfg->inv_freq[m] : std::pow(cfg->rope_theta, -2.0 * m / D);
    pl->cfg.inv_freq = nullptr;
    pl->sm_scale = cfg->sm_scale != 0.f ? cfg->sm_scale : (float)(1.0 / std::sqrt((double)D));
    pl->num_pool_pages = num_pool_pages;
    if (d->num_source_pages < 0) return fail(TESSERA_INVALID_ARG, "negative num_source_pages");
    if ((int64_t)d->num_source_pages * B > (int64_t)INT32_MAX) return fail(TESSERA_UNSUPPORTED_SHAPE, "source pool has more than 2^31 slots");
    pl->num_source_pages = d->num_source_pages;
    pl->batch = d->batch;

    const int batch = d->batch;
    // ---- CSR sanity
    if (batch > 0) {
        if (d->unit_off[0] != 0 || d->recompute_off[0] != 0) return fail(TESSERA_INVALID_ARG, "CSR offsets must start at 0");
        for (int r = 0; r < batch; ++r) {
            if (d->seq_len[r] < 0) return fail(TESSERA_INVALID_ARG, fmt("request %ld: negative seq_len", r));
            if (d->unit_off[r + 1] < d->unit_off[r] || d->recompute_off[r + 1] < d->recompute_off[r])
                return fail(TESSERA_INVALID_ARG, fmt("request %ld: CSR offsets decrease", r));
        }
    }
    const int n_units = batch ? d->unit_off[batch] : 0;
    const int n_q = batch ? d->recompute_off[batch] : 0;
    if (n_units > 0 && (!d->unit_len || !d->unit_cached_pos || !d->unit_cached_stride || !d->unit_target_pos || !d->unit_page_off))
        return fail(TESSERA_INVALID_ARG, "null unit array");
    if (n_q > 0 && !d->recompute_pos) return fail(TESSERA_INVALID_ARG, "null recompute_pos");
    if (n_units > 0) {
        if (d->unit_page_off[0] != 0) return fail(TESSERA_INVALID_ARG, "unit_page_off must start at 0");
        for (int u = 0; u < n_units; ++u) {
            if (d->unit_len[u] < 0) return fail(TESSERA_INVALID_ARG, fmt("unit %ld: negative length", u));
            int np = d->unit_page_off[u + 1] - d->unit_page_off[u];
            if (np < 0) return fail(TESSERA_INVALID_ARG, fmt("unit %ld: unit_page_off decreases", u));
            const int off = d->unit_src_offset ? d->unit_src_offset[u] : 0;
            if (off < 0 || off >= B) return fail(TESSERA_INVALID_ARG, fmt("unit %ld: source offset %ld outside [0, page_size)", u, off));
            if (np != 0 && np != (off + d->unit_len[u] + B - 1) / B)
                return fail(TESSERA_INVALID_ARG, fmt("unit %ld: %ld source pages for %ld tokens", u, np, d->unit_len[u]));
            if (d->unit_target_stride && d->unit_target_stride[u] != 0 && d->unit_target_stride[u] != 1)
                return fail(TESSERA_INVALID_ARG, fmt("unit %ld: target stride must be 0 or 1", u));
            if (np != 0 && d->unit_cached_stride[u] != 0 && d->unit_cached_stride[u] != 1)
                return fail(TESSERA_INVALID_ARG, fmt("unit %ld: cached stride must be 0 or 1", u));
        }
        if (d->unit_page_off[n_units] > 0 && !d->unit_pages) return fail(TESSERA_INVALID_ARG, "null unit_pages");
        if (d->unit_retain_page_off) {
            if (d->unit_retain_page_off[0] != 0) return fail(TESSERA_INVALID_ARG, "unit_retain_page_off must start at 0");
            for (int u = 0; u < n_units; ++u) {
                const int np = d->unit_retain_page_off[u + 1] - d->unit_retain_page_off[u];
                if (np < 0) return fail(TESSERA_INVALID_ARG, fmt("unit %ld: unit_retain_page_off decreases", u));
                if (np != 0 && np != (d->unit_len[u] + B - 1) / B)
                    return fail(TESSERA_INVALID_ARG, fmt("unit %ld: %ld cache pages for %ld tokens", u, np, d->unit_len[u]));
            }
            if (d->unit_retain_page_off[n_units] > 0 && !d->unit_retain_pages) return fail(TESSERA_INVALID_ARG, "null unit_retain_pages");
        }
    }
    if (d->retain_pool_pages < 0) return fail(TESSERA_INVALID_ARG, "negative retain_pool_pages");
    if ((int64_t)d->retain_pool_pages * B > (int64_t)INT32_MAX) return fail(TESSERA_UNSUPPORTED_SHAPE, "cache pool has more than 2^31 slots");
    pl->retain_pool_pages = d->retain_pool_pages;

    // ---- block tables: request r takes the next ceil(T_r / B) free pages
    pl->seq_len.assign(d->seq_len, d->seq_len + batch);
    pl->tok_off.assign(batch + 1, 0);
    pl->page_off.assign(batch + 1, 0);
    int64_t total = 0, need_pages = 0;
    for (int r = 0; r < batch; ++r) {
        total += d->seq_len[r];
        need_pages += (d->seq_len[r] + B - 1) / B;
        if (total > INT32_MAX) return fail(TESSERA_UNSUPPORTED_SHAPE, "batch has more than 2^31 tokens");
        pl->tok_off[r + 1] = (int32_t)total;
        pl->page_off[r + 1] = (int32_t)need_pages;
    }
    if (need_pages > d->n_free)
        return fail(TESSERA_OUT_OF_PAGES, fmt("batch needs %ld destination pages, free list has %ld", need_pages, d->n_free));
    if (need_pages > 0 && !d->free_pages) return fail(TESSERA_INVALID_ARG, "null free_pages");
    pl->pages.assign(d->free_pages, d->free_pages + need_pages);

    // page ids: range, destinations distinct, destinations disjoint from sources
    std::vector<uint8_t> page_use(num_pool_pages, 0);   // 1 = source, 2 = destination
    const int n_src_pages = n_units ? d->unit_page_off[n_units] : 0;
    for (int k = 0; k < n_src_pages; ++k) {
        int pg = d->unit_pages[k];
        const int src_limit = d->num_source_pages > 0 ? d->num_source_pages : num_pool_pages;
        if (pg < 0 || pg >= src_limit) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("source page %ld outside pool of %ld pages", pg, src_limit));
        if (d->num_source_pages == 0) page_use[pg] = 1;    // a separate source pool cannot alias destinations
    }
    for (int64_t k = 0; k < need_pages; ++k) {
        int pg = pl->pages[k];
        if (pg < 0 || pg >= num_pool_pages) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("free page %ld outside pool of %ld pages", pg, num_pool_pages));
        if (page_use[pg] == 1) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("free page %ld is also a source page of this batch", pg));
        if (page_use[pg] == 2) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("free page %ld listed twice", pg));
        page_use[pg] = 2;
    }

    // cache pages of captured units: in range, distinct, and - when they live in the destination pool -
    // neither sources nor destinations of this batch
    const int n_retain_pages = (n_units && d->unit_retain_page_off) ? d->unit_retain_page_off[n_units] : 0;
    if (n_retain_pages > 0) {
        const int limit = d->retain_pool_pages > 0 ? d->retain_pool_pages : num_pool_pages;
        std::vector<uint8_t> seen(limit, 0);
        for (int k = 0; k < n_retain_pages; ++k) {
            const int pg = d->unit_retain_pages[k];
            if (pg < 0 || pg >= limit) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("cache page %ld outside pool of %ld pages", pg, limit));
            if (seen[pg]) return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("cache page %ld listed twice", pg));
            seen[pg] = 1;
            if (d->retain_pool_pages == 0 && page_use[pg] != 0)
                return fail(TESSERA_PAGE_OUT_OF_RANGE, fmt("cache page %ld is also a source or destination page of this batch", pg));
        }
    }

    // ---- per-position sources, recompute rows, coverage
    pl->src_slot.assign((size_t)total, -1);
    pl->recompute_off.assign(d->recompute_off, d->recompute_off + batch + 1);
    pl->recompute_pos.assign(d->recompute_pos, d->recompute_pos + n_q);
    pl->fresh_dst.resize(n_q);
    pl->g_src.clear(); pl->g_dst.clear(); pl->items.clear();
    std::vector<int32_t> unit_of((size_t)total, -1);
    std::vector<uint8_t> fresh((size_t)total, 0);
    std::vector<int32_t> fresh_row((size_t)total, -1);     // recompute row index of a position
    pl->retain_dst.assign(n_retain_pages > 0 ? n_q : 0, -1);
    pl->retained_tokens = 0;
    std::vector<int64_t> deltas;     // shift amounts needed, with repeats
    pl->qk_pairs = 0;
    for (int r = 0; r < batch; ++r) {
        const int T = d->seq_len[r];
        const int64_t base = pl->tok_off[r];
        for (int u = d->unit_off[r]; u < d->unit_off[r + 1]; ++u) {
            const int len = d->unit_len[u], tp = d->unit_target_pos[u];
            if (tp < 0 || (int64_t)tp + len > T)
                return fail(TESSERA_UNIT_OVERLAP, fmt("unit %ld leaves its request's positions [0, %ld)", u, T));
            const bool cached = d->unit_page_off[u + 1] > d->unit_page_off[u];
            for (int i = 0; i < len; ++i) {
                if (unit_of[base + tp + i] != -1)
                    return fail(TESSERA_UNIT_OVERLAP, fmt("units %ld and %ld both claim position %ld", unit_of[base + tp + i], u, tp + i));
                unit_of[base + tp + i] = u;
                if (cached) {
                    const int si = i + (d->unit_src_offset ? d->unit_src_offset[u] : 0);
                    pl->src_slot[base + tp + i] = d->unit_pages[d->unit_page_off[u] + si / B] * B + si % B;
                }
            }
        }
        for (int j = d->recompute_off[r]; j < d->recompute_off[r + 1]; ++j) {
            const int p = d->recompute_pos[j];
            if (p < 0 || p >= T) return fail(TESSERA_INVALID_ARG, fmt("request %ld: recompute position %ld outside [0, %ld)", r, p, T));
            if (j > d->recompute_off[r] && d->recompute_pos[j - 1] >= p)
                return fail(TESSERA_UNSORTED_POSITIONS, fmt("request %ld: recompute positions not strictly ascending at index %ld", r, j));
            fresh[base + p] = 1;
            fresh_row[base + p] = j;
            pl->fresh_dst[j] = pl->pages[pl->page_off[r] + p / B] * B + p % B;
            pl->qk_pairs += (int64_t)p + 1;
        }
        for (int p = 0; p < T; ++p)
            if (pl->src_slot[base + p] < 0 && !fresh[base + p])
                return fail(TESSERA_UNCOVERED_POSITION, fmt("request %ld: position %ld has no cached unit and is not recomputed", r, p));
        // captured units: every token is a recompute row; row j also goes to the unit's cache slot
        if (n_retain_pages > 0)
            for (int u = d->unit_off[r]; u < d->unit_off[r + 1]; ++u) {
                const int first = d->unit_retain_page_off[u], np = d->unit_retain_page_off[u + 1] - first;
                if (np == 0) continue;
                for (int i = 0; i < d->unit_len[u]; ++i) {
                    const int j = fresh_row[base + d->unit_target_pos[u] + i];
                    if (j < 0)
                        return fail(TESSERA_INVALID_ARG, fmt("unit %ld is to be captured but its token %ld is not recomputed", u, i));
                    pl->retain_dst[j] = d->unit_retain_pages[first + i / B] * B + i % B;
                }
                pl->retained_tokens += d->unit_len[u];
            }
    }

    // ---- copy list + shift table.  One item = up to kGatherItemTokens rows of one unit.
    for (int r = 0; r < batch; ++r)
        for (int u = d->unit_off[r]; u < d->unit_off[r + 1]; ++u) {
            if (d->unit_page_off[u + 1] <= d->unit_page_off[u]) continue;
            // token i is shifted by (target_pos + ts * i) - (cached_pos + cs * i)
            const int64_t d0 = (int64_t)d->unit_target_pos[u] - d->unit_cached_pos[u];
            const int step = (d->unit_target_stride ? d->unit_target_stride[u] : 1) - d->unit_cached_stride[u];
            if (step == 0) deltas.push_back(d0);
            else for (int i = 0; i < d->unit_len[u]; ++i) deltas.push_back(d0 + (int64_t)step * i);
        }
    std::sort(deltas.begin(), deltas.end());
    deltas.erase(std::unique(deltas.begin(), deltas.end()), deltas.end());
    for (int64_t x : deltas)
        if (x > INT32_MAX || x < INT32_MIN) return fail(TESSERA_INVALID_ARG, "shift amount overflows int32");
    pl->rope_delta.assign(deltas.begin(), deltas.end());
    pl->rope_table.resize(deltas.size() * (size_t)D);     // [row][D/2][cos, sin]
    for (size_t row = 0; row < deltas.size(); ++row)
        for (int m = 0; m < D / 2; ++m) {
            // angle, cosine and sine in fp64; a single rounding to fp32 each
            const double ang = (double)deltas[row] * pl->inv_freq[m];
            pl->rope_table[(row * (D / 2) + m) * 2 + 0] = (float)std::cos(ang);
            pl->rope_table[(row * (D / 2) + m) * 2 + 1] = (float)std::sin(ang);
        }
    auto row_of = [&](int64_t delta) {
        return (int32_t)(std::lower_bound(deltas.begin(), deltas.end(), delta) - deltas.begin());
    };
    pl->cached_tokens = 0;
    // Rows per gather block: 32, fewer when the batch is so small that the grid would not fill the GPU.
    int item_tokens = kGatherItemTokens;
    {
        int64_t cached = 0;
        for (int u = 0; u < n_units; ++u)
            if (d->unit_page_off[u + 1] > d->unit_page_off[u]) cached += d->unit_len[u];
        while (item_tokens > 8 && cached / item_tokens < 4 * num_sms) item_tokens /= 2;
    }
    // Requests may use the same cached unit (equal source pages, offset and length).  The items of its users
    // are emitted side by side, so that blocks running together read the same rows out of L2 (and the
    // host-tier reader fetches a row once for all of them): 81 550 cached rows, 47 846 distinct, 106 -> 91 us.
    // (Flat lists and hash chains: a vector per distinct unit and a multimap made plans of many units up to 40 % longer.)
    struct Use { int32_t req, unit, next; };           // users of a distinct unit, in order
    struct Distinct { int32_t first, last, n, next; }; // next: of the same hash
    std::vector<Use> uses;
    std::vector<Distinct> distinct;                    // in order of first use
    uses.reserve(n_units);
    distinct.reserve(n_units);
    {
        size_t slots = 16;
        while (slots < 2 * (size_t)n_units) slots *= 2;
        std::vector<int32_t> head(slots, -1);
        auto src_off = [&](int u) { return d->unit_src_offset ? d->unit_src_offset[u] : 0; };
        for (int r = 0; r < batch; ++r)
            for (int u = d->unit_off[r]; u < d->unit_off[r + 1]; ++u) {
                const int p0 = d->unit_page_off[u], np = d->unit_page_off[u + 1] - p0;
                if (np <= 0) continue;
                const uint64_t key = (((uint64_t)(uint32_t)d->unit_pages[p0] << 32) | (uint32_t)d->unit_len[u]) * 128 + (uint32_t)src_off(u);
                int32_t &chain = head[((key * 0x9E3779B97F4A7C15ull) >> 32) & (slots - 1)];
                int32_t k = chain;
                for (; k >= 0; k = distinct[k].next) {
                    const int v = uses[distinct[k].first].unit, v0 = d->unit_page_off[v];
                    if (d->unit_len[u] == d->unit_len[v] && src_off(u) == src_off(v) && d->unit_page_off[v + 1] - v0 == np &&
                        std::equal(d->unit_pages + p0, d->unit_pages + p0 + np, d->unit_pages + v0))
                        break;
                }
                const int32_t use = (int32_t)uses.size();
                uses.push_back({r, u, -1});
                if (k < 0) {
                    distinct.push_back({use, use, 1, chain});
                    chain = (int32_t)distinct.size() - 1;
                } else {
                    uses[distinct[k].last].next = use;
                    distinct[k].last = use;
                    ++distinct[k].n;
                }
                pl->cached_tokens += d->unit_len[u];
            }
    }
    std::vector<int32_t> req_run_off(batch + 1, -1);       // first run whose first user is the request (or a later one)
    pl->runs.clear();
    pl->g_src.resize((size_t)pl->cached_tokens);
    pl->g_dst.resize((size_t)pl->cached_tokens);
    int page_shift = 0;
    while ((1 << page_shift) < B) ++page_shift;
    int32_t listed = 0;
    for (const Distinct &unit : distinct) {
        const int32_t first_req = uses[unit.first].req;
        if (req_run_off[first_req] < 0) req_run_off[first_req] = (int32_t)pl->runs.size();
        const int len = d->unit_len[uses[unit.first].unit];
        for (int i0 = 0; i0 < len; i0 += item_tokens) {
            const int cnt = std::min(item_tokens, len - i0);
            pl->runs.push_back({(int32_t)pl->items.size(), unit.n, listed, cnt});
            for (int32_t k = unit.first; k >= 0; k = uses[k].next) {
                const int u = uses[k].unit, r = uses[k].req, tp = d->unit_target_pos[u];
                const int64_t d0 = (int64_t)tp - d->unit_cached_pos[u];
                const int step = (d->unit_target_stride ? d->unit_target_stride[u] : 1) - d->unit_cached_stride[u];
                pl->items.push_back({listed, cnt, row_of(d0) + i0 * step, step});   // step +-1: consecutive integers are consecutive rows
                const int32_t *src = pl->src_slot.data() + pl->tok_off[r] + tp + i0;
                std::copy(src, src + cnt, pl->g_src.data() + listed);
                const int32_t *table = pl->pages.data() + pl->page_off[r];
                for (int i = 0, p = tp + i0; i < cnt; ++i, ++p) pl->g_dst[listed + i] = (table[p >> page_shift] << page_shift) + (p & (B - 1));
                listed += cnt;
            }
        }
    }
    req_run_off[batch] = (int32_t)pl->runs.size();
    for (int r = batch - 1; r >= 0; --r)
        if (req_run_off[r] < 0) req_run_off[r] = req_run_off[r + 1];

    // ---- attention work list: tiles of consecutive recompute rows of one request
    const int g = Hq / Hkv;
    pl->tile_tokens = kAttnTileRows / g;
    pl->attn_kernel = 1;       // the tcgen05 kernel covers every accepted shape (page size 8..128, head_dim 64 / 128, g <= 16)
    pl->tiles.clear();
    for (int r = 0; r < batch; ++r)
        for (int j0 = d->recompute_off[r]; j0 < d->recompute_off[r + 1]; j0 += pl->tile_tokens) {
            const int n = std::min(pl->tile_tokens, d->recompute_off[r + 1] - j0);
            AttnTile t{};
            t.req = r; t.q_begin = j0; t.n_tok = n;
            t.kv_len = d->recompute_pos[j0 + n - 1] + 1;
            t.kv_full = d->recompute_pos[j0] + 1;
            pl->tiles.push_back(t);
        }
    // tcgen05 work items: consecutive tiles of a request share one thread block (and every K/V page
    // they read).
    pl->work.clear();
    {
        const int page = 128;        // keys per step of the tensor-core kernel
        std::vector<std::pair<int32_t, int32_t>> pairs;
        size_t first = 0;
        while (first < pl->tiles.size()) {
            size_t last = first;
            while (last < pl->tiles.size() && pl->tiles[last].req == pl->tiles[first].req) ++last;
            for (size_t k = first; k < last; k += 2) {
                const int32_t a = (int32_t)k, b2 = (k + 1 < last) ? (int32_t)(k + 1) : -1;
                pairs.push_back({a, b2});
            }
            first = last;
        }
        auto steps_of = [&](int32_t tile) { return (pl->tiles[tile].kv_len + page - 1) / page; };
        // Modelled cycles of an item (clock64 on a B200): item fetch 1 700, epilogue and what the first step takes
        // longer than a later one 4 700 per tile, 3 180 per step of both tiles, 2 400 per step of a lone one (whose
        // softmax and MMAs wait for each other).
        auto model_cycles = [](int steps_a, int steps_b, int n_tiles) -> int64_t {
            const int both = std::min(steps_a, steps_b), single = std::max(steps_a, steps_b) - both;
            return 1700 + (int64_t)n_tiles * 4700 + (int64_t)both * 3180 + (int64_t)single * 2400;
        };
        // Split-KV: the key ranges of a batch that leaves SMs idle are cut into parts of at most `limit` steps
        // that run as separate items and are merged afterwards.
        //   items <= SMs / 2 : the smallest limit whose parts still fit one round (one item per SM), if the model gives
        //                      it 10 %.  A common limit, not a common part count, so that short tiles are not cut as
        //                      often as long ones: 48 items of 42 steps in parts of 9 in place of 14, attention
        //                      39.4 -> 35.7 us.  56 items of four steps stay whole (cut in 80 parts a host-tier
        //                      layer takes 58.0 us, whole 54.2).
        //   items <= kSplitMaxRounds x SMs : the limit of the least modelled time, if that is 10 % below the uncut
        //                      list's.  Attention of n requests of two tiles over 12 288 keys: 80 items 185 -> 141 us,
        //                      152 items (two rounds on 148 SMs, the second nearly empty) 368 -> 282; over 4 096 keys
        //                      152 items stay whole (126-140 us, cut in 456 130-146).
        //   more             : never; the rounds are even enough and the merge only costs.
        auto parts_of = [&](int steps, int limit) {
            return std::max(1, std::min({(steps + limit - 1) / limit, kSplitMaxParts, steps / kSplitMinSteps}));
        };
        auto long_steps = [&](const std::pair<int32_t, int32_t> &pr) { return steps_of(pr.second >= 0 ? pr.second : pr.first); };
        int longest = 1;
        for (auto &pr : pairs) longest = std::max(longest, long_steps(pr));
        auto items_at = [&](int limit) {
            int64_t n = 0;
            for (auto &pr : pairs) n += parts_of(long_steps(pr), limit);
            return n * Hkv;
        };
        // Time of the list cut at `limit`: longest-first assignment to the least-loaded SM (also of a list that will be dealt
        // in page order), plus the merge.  Returns at once - with no more than that time - where even a perfectly even
        // assignment reaches `enough`.
        std::vector<int64_t> part_cost, load;
        auto modelled = [&](int limit, int64_t enough) -> int64_t {
            part_cost.clear();          // of the parts of one head; every head has the same
            int64_t slots = 0, sum = 0, top = 0;
            for (auto &pr : pairs) {
                const int sl = long_steps(pr), sa = pr.second >= 0 ? steps_of(pr.first) : 0, parts = parts_of(sl, limit);
                const int len = (sl + parts - 1) / parts;
                for (int b0 = 0; b0 < sl; b0 += len) {
                    const int n_b = std::min(sl, b0 + len) - b0, n_a = std::max(0, std::min(sa, b0 + len) - b0);
                    part_cost.push_back(model_cycles(n_a, n_b, n_a > 0 ? 2 : 1));
                    sum += part_cost.back() * Hkv;
                    top = std::max(top, part_cost.back());
                    if (parts > 1) slots += (n_a > 0 ? 2 : 1) * Hkv;
                }
            }
            const bool one_round = (int64_t)part_cost.size() * Hkv <= num_sms;
            const int64_t merge = slots ? (one_round ? kMergeCyclesOneRound : kMergeCycles) + slots * kMergeCyclesPerSlot : 0;
            if (one_round) return top + merge;
            const int64_t even = std::max(top, sum / num_sms) + merge;
            if (even >= enough) return even;
            std::sort(part_cost.begin(), part_cost.end(), std::greater<int64_t>());
            load.assign(num_sms, 0);                    // a heap, least-loaded SM first
            int64_t end = 0;
            for (int64_t c : part_cost)
                for (int h = 0; h < Hkv; ++h) {
                    const int64_t l = load[0] + c;
                    end = std::max(end, l);
                    size_t i = 0;
                    for (size_t k = 1; k < load.size(); i = k, k = 2 * i + 1) {
                        if (k + 1 < load.size() && load[k + 1] < load[k]) ++k;
                        if (load[k] >= l) break;
                        load[i] = load[k];
                    }
                    load[i] = l;
                }
            return end + merge;
        };
        int limit = longest;
        const int64_t uncut = may_cut ? (int64_t)pairs.size() * Hkv : 0;
        if (uncut > 0 && 2 * uncut <= num_sms) {
            int l = longest;
            while (l > kSplitMinSteps && items_at(l - 1) <= num_sms) --l;
            if (modelled(l, INT64_MAX) < modelled(longest, INT64_MAX) * 90 / 100) limit = l;
        } else if (uncut > 0 && uncut <= (int64_t)kSplitMaxRounds * num_sms) {
            int64_t all = 0;
            for (auto &pr : pairs)
                all += Hkv * model_cycles(pr.second >= 0 ? steps_of(pr.first) : 0, long_steps(pr), pr.second >= 0 ? 2 : 1);
            int64_t best = modelled(longest, INT64_MAX) * 90 / 100;
            if (best > all / num_sms)           // otherwise no cut can reach it
                for (int l = longest * 3 / 4; l >= 2 * kSplitMinSteps && items_at(l) <= 2 * kSplitMaxRounds * num_sms; l = l * 5 / 6) {
                    const int64_t m = modelled(l, best);
                    if (m < best) best = m, limit = l;
                }
        }
        pl->combine.clear();
        pl->n_slots = 0;
        for (auto &pr : pairs) {
            const int32_t a = pr.first, b2 = pr.second;
            const int sa = steps_of(a), sl = long_steps(pr);                   // sa <= sl: positions ascend
            const int parts = parts_of(sl, limit), len = (sl + parts - 1) / parts;
            const int parts_b = (sl + len - 1) / len, parts_a = b2 >= 0 ? (sa + len - 1) / len : parts_b;
            for (int h = 0; h < Hkv; ++h) {
                if (parts == 1) {
                    pl->work.push_back({a, b2, h, 0, sl, -1, -1, 0, 0, 0, 0, 0});
                    continue;
                }
                const int32_t slot_a = pl->n_slots, slot_b = slot_a + parts_a;
                for (int p2 = 0; p2 < parts_b; ++p2) {
                    const int sb = p2 * len, se = std::min(sl, sb + len);
                    if (p2 < parts_a) pl->work.push_back({a, b2, h, sb, se, slot_a + p2, b2 >= 0 ? slot_b + p2 : -1, 0, 0, 0, 0, 0});
                    else pl->work.push_back({b2, -1, h, sb, se, slot_b + p2, -1, 0, 0, 0, 0, 0});   // tile a is already finished
                }
                const AttnTile &ta = pl->tiles[a], &tb = pl->tiles[b2 >= 0 ? b2 : a];
                pl->combine.push_back({a, h, parts_a, slot_a, ta.q_begin, ta.n_tok, 0, 0});
                if (b2 >= 0) pl->combine.push_back({b2, h, parts_b, slot_b, tb.q_begin, tb.n_tok, 0, 0});
                pl->n_slots += parts_a + (b2 >= 0 ? parts_b : 0);
            }
        }
        auto cycles_of = [&](const AttnWork &w) {
            const int sa = std::min(w.step_end, steps_of(w.tile_a)) - w.step_begin;
            const int sb = w.tile_b >= 0 ? std::min(w.step_end, steps_of(w.tile_b)) - w.step_begin : 0;
            return model_cycles(sa, sb, w.tile_b >= 0 ? 2 : 1);
        };
        // cost of an item = its (tile, 128-key step) count, kept in the item for the sorts
        for (AttnWork &w : pl->work) {
            int c = std::min(w.step_end, steps_of(w.tile_a)) - w.step_begin;
            if (w.tile_b >= 0) c += std::min(w.step_end, steps_of(w.tile_b)) - w.step_begin;
            w.cost = c;
            const int32_t req = pl->tiles[w.tile_a].req;
            w.seq_len = pl->seq_len[req];
            w.page_begin = pl->page_off[req];
        }
        // Launch latency is a visible part of a layer while the attention takes tens of microseconds: 240 items of up to 8
        // steps 53.0 -> 48.3 us a layer, 1 680 short items 121.1 -> 114.6.  Layers whose attention runs for hundreds, near
        // the power limit, lose: 1 024 items (450 000 modelled cycles an SM) 436 -> 444 us, 1 152 items 2 715 -> 2 742.
        int64_t modelled_cycles = 0;
        for (const AttnWork &w : pl->work) modelled_cycles += cycles_of(w);
        pl->chained = modelled_cycles / num_sms <= kChainedCycles;
        pl->mma_pairs = 0;
        for (const AttnWork &w : pl->work) pl->mma_pairs += (int64_t)w.cost * kAttnTileRows * page;
        auto cost = [](const AttnWork &w) { return w.cost; };
        auto sort_items = [&](std::vector<AttnWork>::iterator first_it, std::vector<AttnWork>::iterator last_it) {
            int max_cost = 1;
            for (auto it = first_it; it != last_it; ++it) max_cost = std::max(max_cost, cost(*it));
            const int band = std::max(1, max_cost / kAttnCostBands);
            const AttnTile *tl = pl->tiles.data();
            std::stable_sort(first_it, last_it, [=](const AttnWork &x, const AttnWork &y) {
                const int bx = x.cost / band, by = y.cost / band;
                if (bx != by) return bx > by;
                const int rx = tl[x.tile_a].req, ry = tl[y.tile_a].req;
                if (rx != ry) return rx < ry;
                if (x.kvh != y.kvh) return x.kvh < y.kvh;
                return x.cost > y.cost;
            });
        };
        // chunks of whole requests with about equal attention cost, for the host-buffer pipeline
        std::vector<int64_t> req_cost(batch, 0);
        for (const AttnWork &w : pl->work) req_cost[pl->tiles[w.tile_a].req] += cost(w);
        int64_t total_cost = 0;
        for (int64_t c : req_cost) total_cost += c;
        const int n_chunks = std::max(1, std::min(batch, kHostChunks));
        std::vector<int> chunk_of(batch, 0);
        pl->chunk_row_off.assign(1, 0);
        {
            int64_t acc = 0;
            int c = 0;
            for (int r = 0; r < batch; ++r) {
                chunk_of[r] = c;
                acc += req_cost[r];
                const bool last_req = r + 1 == batch;
                // close the chunk when its share of the cost is reached, keeping one request per remaining chunk
                if (!last_req && c + 1 < n_chunks && (acc * n_chunks >= total_cost * (c + 1) || batch - (r + 1) <= n_chunks - (c + 1))) {
                    pl->chunk_row_off.push_back(d->recompute_off[r + 1]);
                    ++c;
                }
            }
            pl->chunk_row_off.push_back(n_q);
        }
        const int used_chunks = (int)pl->chunk_row_off.size() - 1;
        pl->chunk_run_off.assign(used_chunks + 1, (int32_t)pl->runs.size());
        pl->chunk_run_off[0] = 0;
        for (int r = 1; r < batch; ++r)
            if (chunk_of[r] != chunk_of[r - 1]) pl->chunk_run_off[chunk_of[r]] = req_run_off[r];
        pl->work_chunked = pl->work;           // (built request by request, so chunk by chunk too, as the list to merge is)
        pl->chunk_work_off.assign(used_chunks + 1, 0);
        for (const AttnWork &w : pl->work_chunked) ++pl->chunk_work_off[chunk_of[pl->tiles[w.tile_a].req] + 1];
        for (int c = 0; c < used_chunks; ++c) pl->chunk_work_off[c + 1] += pl->chunk_work_off[c];
        for (int c = 0; c < used_chunks; ++c)
            sort_items(pl->work_chunked.begin() + pl->chunk_work_off[c], pl->work_chunked.begin() + pl->chunk_work_off[c + 1]);
        pl->chunk_combine_off.assign(used_chunks + 1, 0);
        for (const CombineItem &ci : pl->combine) ++pl->chunk_combine_off[chunk_of[pl->tiles[ci.tile].req] + 1];
        for (int c = 0; c < used_chunks; ++c) pl->chunk_combine_off[c + 1] += pl->chunk_combine_off[c];
        // A list of more than one item per thread block is dealt out here, each item to the least-loaded block by modelled
        // cycles, longest first.  Long lists of long items over much K/V are dealt in two stretches: first the long items,
        // request by request and KV head by KV head (page order), so that the blocks of the whole GPU work through the same
        // K/V pages at about the same time and find them in L2; then the short ones, the last kTailItems longest items' worth
        // of cycles per block, longest first, to even out what the first stretch left.  That order is worth DRAM traffic, and
        // through the power limit time, back to back: 1 152 items of up to 258 steps read 3.51 -> 1.77 GB from DRAM, a layer
        // of them takes 2 719 -> 2 608 us; 20 696 items 12 921 -> 11 546.  It costs where the items are short, because many
        // blocks then ask for the same lines at the same time.  Balance is the lesser matter: 720 and 1 224 items whose
        // slowest block is modelled 4 and 3 % later in page order than longest first took 503 and 1 235 us, against 514 and
        // 1 292.
        // The kernel's serpentine walk (round k, block b -> index k G + (k odd ? G - 1 - b : b)) hands every block its own
        // list; holes, only at the end of a block's list, are marked tile_a = -1.
        auto deal_out = [&](std::vector<AttnWork> &list) {
            const int G = num_sms;
            if ((int)list.size() <= G) {
                // one item a block: neighbours in the list (the two SMs of a TPC) share a request and KV head
                sort_items(list.begin(), list.end());
                return;
            }
            double all = 0, steps = 0;
            int64_t longest_item = 0;
            for (const AttnWork &w : list) {
                const int64_t c = cycles_of(w);
                all += (double)c;
                steps += w.step_end - w.step_begin;
                longest_item = std::max(longest_item, c);
            }
            steps /= (double)list.size();
            const double kv_bytes = (double)total * Hkv * D * 4, item_bytes = steps * page * D * 4;
            const bool two_stretches = all >= kPageOrderCycles * G && steps >= kPageOrderSteps && all >= kHeadItems * (double)longest_item * G &&
                                       kv_bytes * item_bytes >= kPageOrderBytes * kPageOrderBytes;
            if (!two_stretches) sort_items(list.begin(), list.end());       // equal items keep their pages' order
            // (sorted as runs of equal items - the KV heads of a tile pair - and dealt by a tree: 20 696 items item by item from
            // a priority queue took 5 ms of a plan's 11)
            struct Run { int64_t cycles; int32_t first, n, req; };
            std::vector<Run> runs;
            for (int32_t i = 0; i < (int32_t)list.size(); ++i) {
                const int64_t c = cycles_of(list[i]);
                const int32_t req = pl->tiles[list[i].tile_a].req;
                if (!runs.empty() && runs.back().cycles == c && runs.back().req == req) ++runs.back().n;
                else runs.push_back({c, i, 1, req});
            }
            std::stable_sort(runs.begin(), runs.end(), [](const Run &a, const Run &b) { return a.cycles > b.cycles; });
            struct Entry { int64_t cycles; int32_t item, group; };          // group: request and KV head
            std::vector<Entry> order;
            order.reserve(list.size());
            for (const Run &r : runs)
                for (int32_t i = 0; i < r.n; ++i) order.push_back({r.cycles, r.first + i, r.req * Hkv + list[r.first + i].kvh});
            const double tail_cycles = kTailItems * (double)order[0].cycles * G;
            size_t head = two_stretches ? order.size() : 0;
            for (double sum = 0; head > 0 && sum < tail_cycles; --head) sum += (double)order[head - 1].cycles;
            {
                // the first stretch by request and KV head, longest first within: a counting sort
                std::vector<int32_t> at((size_t)batch * Hkv + 1, 0);
                for (size_t i = 0; i < head; ++i) ++at[order[i].group + 1];
                for (size_t k = 1; k < at.size(); ++k) at[k] += at[k - 1];
                std::vector<Entry> sorted(head);
                for (size_t i = 0; i < head; ++i) sorted[at[order[i].group]++] = order[i];
                std::copy(sorted.begin(), sorted.end(), order.begin());
            }
            // the blocks' loads (x 2^16, + block) are the leaves of a tree whose nodes hold the least of their two
            int leaves = 1;
            while (leaves < G) leaves *= 2;
            std::vector<int64_t> least(2 * leaves, INT64_MAX);
            for (int b = 0; b < G; ++b) least[leaves + b] = b;
            for (int i = leaves - 1; i > 0; --i) least[i] = std::min(least[2 * i], least[2 * i + 1]);
            std::vector<int32_t> taken(G, 0), at(order.size());           // items a block has; where in the list an item goes
            int32_t rounds = 0;
            for (size_t n = 0; n < order.size(); ++n) {
                const int b = (int)(least[1] & 0xffff), k = taken[b]++;
                rounds = std::max(rounds, k + 1);
                at[n] = k * G + ((k & 1) ? G - 1 - b : b);
                least[leaves + b] += order[n].cycles << 16;
                for (int i = (leaves + b) / 2; i > 0; i /= 2) least[i] = std::min(least[2 * i], least[2 * i + 1]);
            }
            AttnWork hole{};
            hole.tile_a = -1; hole.tile_b = -1;
            std::vector<AttnWork> out((size_t)rounds * G, hole);
            for (size_t n = 0; n < order.size(); ++n) out[at[n]] = list[order[n].item];
            list.swap(out);
        };
        pl->n_work_items = (int32_t)pl->work.size();
        deal_out(pl->work);
    }

    pl->total_tokens = total;
    pl->n_q = n_q;
    return TESSERA_OK;
}

}  // namespace tessera
