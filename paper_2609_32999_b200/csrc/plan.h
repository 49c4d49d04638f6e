// Internal plan representation shared by the host builder and the launch code.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>
#include <vector_types.h>

#include "blob_pool.h"
#include "tessera.h"

namespace tessera {

constexpr int kGatherItemTokens = 32;   // token rows per thread block of the gather kernel
constexpr int kAttnTileRows = 128;      // query rows (tokens x grouped heads) per tcgen05 tile
constexpr int kDefaultSMs = 148;         // SM count assumed by a host-only plan (a B200); device plans ask the device
constexpr int kSplitMinSteps = 2;        // never split below this many 128-key steps per part
constexpr int kSplitMaxParts = 32;
constexpr int kChainedCycles = 300000;   // modelled attention cycles per SM up to which launches are chained
constexpr int kSplitMaxRounds = 4;       // batches of more attention items per SM than this are never split, and a split
                                         // list has at most twice as many parts (each with up to two workspace slots)
constexpr int kHostChunks = 4;          // request chunks of the host-buffer entry point's copy / compute pipeline
// An attention list is dealt out in page order first (see build_plan_host) where, modelled and averaged over the list, ...
constexpr double kPageOrderCycles = 225000;   // ... an SM has this many cycles of it and more, so that calls back to back reach the power limit:
                                              // 9 to 12 steps an item, 130-220 000 cycles 1-3 % slower in page order, 230-260 000 3 % faster
constexpr double kPageOrderSteps = 9;         // ... an item has this many 128-key steps: 3-5 steps 8-20 % slower (over 285 MB and more of K/V),
                                              // 7-8 5 % slower to 4 % faster, 9.2 2.8 % faster, 17-21 4-8 %, 33 and more 4-13 %
constexpr double kPageOrderBytes = 8.4e6;     // ... and this is at most the geometric mean of what an item reads (64 KB a step at head_dim 128)
                                              // and the batch's K/V: 12 steps, 75 MB (7.7e6) 2.7 % slower; 10.6, 131 (9.5e6) 0.3 %; 12.6, 88
                                              // (8.5e6) and 13, 120 (10e6) 2.2 and 3.6 % faster; 42, 35 (9.8e6) 1.6 %; at head_dim 64 14.5, 78
                                              // (6.1e6) 3.8 % slower; 26, 83 (8.4e6) 0.9 %; 17, 138 (8.8e6) 1.4 % faster.  From 17e6 on 3-13 %.
constexpr double kHeadItems = 2.5;       // ... it has this much work per block, in longest items (2.1: 2 % slower; 2.6, 3.6 and 4.3: 3-4 % faster)
constexpr double kTailItems = 0.6;       // work kept back to even out the blocks, in longest items per block (0.3: up to 13 % slower, 0.9 and
                                         // 1.3: 1-4 % slower on lists of 7 to 140 items per block)
constexpr int kAttnCostBands = 16;      // cost bands (longest band first) of a list of one item a block or of a chunk; elsewhere the order of equal items

// One thread block of the gather / shift kernel: `count` consecutive entries of the copy list that
// belong to one cached unit.  Entry i uses row (row0 + i * row_step) of the cos/sin table.
struct GatherItem {
    int32_t begin, count, row0, row_step;
};

// One source run of the host-tier reader: gather items [first_item, first_item + n_items) read the same
// rows of the same cached unit (one item per request that uses it) and differ only in slots and shifts.
struct GatherRun {
    int32_t first_item, n_items;
    int32_t begin, count;      // of the first item: its source rows are everyone's
};

// One query tile of the attention kernel: `n_tok` consecutive recompute rows [q_begin, q_begin+n_tok)
// of request `req`; the tile reads keys [0, kv_len).  Keys below `kv_full` are visible to every row.
struct AttnTile {
    int32_t req, q_begin, n_tok, kv_len, kv_full, pad0, pad1, pad2;
};

// One thread block of the tcgen05 attention kernel: KV head `kvh` of query tiles tile_a and tile_b
// (consecutive tiles of one request; tile_b = -1 when the request has an odd tile left over).
// With split-KV the item covers only the 128-key steps [step_begin, step_end) and leaves its tiles' partial
// results in workspace slots slot_a / slot_b (-1: the item covers the whole key range of its tiles and writes
// the outputs); a part in which tile_a would have nothing to do names the longer tile alone.
struct AttnWork {
    int32_t tile_a, tile_b, kvh, step_begin, step_end, slot_a, slot_b;
    int32_t cost;      // (tile, step) count of the item: the host's sort key, not read by the kernel
    int32_t seq_len, page_begin;   // of the request: its length and first block-table entry (so that the loads of K and V
                                   // wait for this record and the page ids only, not for a chain through the tiles)
    int32_t pad0, pad1;
};

// One (query tile, KV head) whose partial results have to be merged after a split-KV launch.
struct CombineItem {
    int32_t tile, kvh, n_parts, slot0;   // partial results in workspace slots [slot0, slot0 + n_parts)
    int32_t q_begin, n_tok;              // of the tile
    int32_t pad0, pad1;
};

struct DeviceTables {
    DeviceBlob blob;               // one allocation holding everything below
    int32_t *g_src = nullptr, *g_dst = nullptr;
    GatherItem *items = nullptr;
    GatherRun *runs = nullptr;
    float2 *rope = nullptr;        // [n_rope_rows][D/2] (cos, sin)
    int32_t *fresh_dst = nullptr;  // [n_q] destination slot of each recompute row
    int32_t *retain_dst = nullptr; // [n_q] cache slot of a captured row, -1 otherwise (null: nothing is captured)
    int32_t *q_pos = nullptr;      // [n_q]
    int32_t *pages = nullptr;      // block tables
    AttnTile *tiles = nullptr;
    AttnWork *work = nullptr;      // tcgen05 work items, dealt out to the thread blocks
    AttnWork *work_chunked = nullptr;  // the same items grouped by request chunk, longest first (host-buffer entry)
    CombineItem *combine = nullptr;    // (tile, head) pairs to merge, grouped by request chunk
    float *ws_o = nullptr;             // split-KV partials: [slot][16 rows][8 columns][lane][4] unnormalised O ...
    float2 *ws_ml = nullptr;           // ... and [slot][128] (reference maximum in log2 units, sum)
    int32_t *status = nullptr;     // device status word(s)
    double *inv_freq = nullptr;    // [D/2] rotary frequencies
    DeviceBlob q8;                 // 8-bit copy of q for the 8-bit-key attention entry (allocated on first use)
    DeviceBlob staging;            // of the host-buffer entry point (allocated on first use), holding:
    void *st_q = nullptr, *st_k = nullptr, *st_v = nullptr, *st_o = nullptr;
    float *st_lse = nullptr;
};

}  // namespace tessera

struct tessera_plan {
    tessera_model_cfg cfg{};
    std::vector<double> inv_freq;          // [D/2], always filled
    float sm_scale = 0.f;
    int32_t num_pool_pages = 0;
    int32_t num_source_pages = 0;          // > 0: cached units are read from a separate source pool
    int32_t batch = 0;
    bool host_only = false;
    int device = -1;
    int num_sms = tessera::kDefaultSMs;    // multiprocessors of the plan's device: grid of the persistent attention
                                           // kernel, target block count of split-KV and of the small-batch gather

    std::vector<int32_t> seq_len, tok_off, page_off, pages, src_slot;
    std::vector<int32_t> recompute_off, recompute_pos, fresh_dst;
    std::vector<int32_t> retain_dst;       // [n_q] or empty: cache slot of every captured recompute row
    int32_t retain_pool_pages = 0;         // > 0: captured units go to a separate cache pool of this many pages
    int64_t retained_tokens = 0;
    std::vector<int32_t> g_src, g_dst;
    std::vector<tessera::GatherItem> items;
    std::vector<tessera::GatherRun> runs;  // the items, grouped by source rows (order of first use)
    std::vector<int32_t> rope_delta;       // sorted distinct shift amounts
    std::vector<float> rope_table;         // [rows][D/2][2]
    std::vector<tessera::AttnTile> tiles;
    std::vector<tessera::AttnWork> work;
    // The host-buffer entry point pipelines copies against compute over chunks of whole requests.
    std::vector<tessera::AttnWork> work_chunked;   // items of chunk c: [chunk_work_off[c], chunk_work_off[c+1])
    std::vector<int32_t> chunk_work_off, chunk_row_off;   // [n_chunks + 1]; rows = recompute rows
    std::vector<int32_t> chunk_run_off;                   // [n_chunks + 1]; gather runs first used by the chunk's requests
    std::vector<tessera::CombineItem> combine;     // grouped by chunk: [chunk_combine_off[c], chunk_combine_off[c+1])
    std::vector<int32_t> chunk_combine_off;
    int32_t n_work_items = 0;                      // real items of `work` (the list may hold holes)
    // Kernels of the plan's calls are launched chained (see launch_kernel): the attention is short.
    bool chained = false;
    int32_t n_slots = 0;                           // split-KV workspace slots (0 = nothing is split)
    int32_t attn_kernel = 0;
    int32_t tile_tokens = 0;

    int64_t total_tokens = 0, n_q = 0, cached_tokens = 0, qk_pairs = 0, mma_pairs = 0;

    std::vector<char> host_blob;           // staging image of the device tables
    tessera::DeviceTables dev;
    // streams / events of the host-buffer entry point (created on first use)
    cudaStream_t s_in = nullptr, s_out = nullptr;
    cudaEvent_t ev_start = nullptr, ev_out = nullptr;
    std::vector<cudaEvent_t> ev_in, ev_comp;
};

namespace tessera {
// Builds and validates all host tables.  Returns a status; on failure `err` holds the reason.
// `num_sms`: multiprocessor count the work lists are sized for.  `may_cut`: key ranges may be cut (split-KV).
int32_t build_plan_host(const tessera_model_cfg *cfg, const tessera_compose_desc *desc,
                        int32_t num_pool_pages, int num_sms, bool may_cut, tessera_plan *plan, std::string *err);

// Thread blocks of an attention launch over the whole list (chunk < 0) or a chunk's: one per SM, `max_blocks` > 0 at most,
// no more than items.  0 where the list cannot be walked by so few: a dealt list has holes that end a block's share only
// on the grid it was dealt for.
inline int attn_grid(const tessera_plan *pl, int chunk, int max_blocks) {
    const size_t n = chunk < 0 ? pl->work.size() : (size_t)(pl->chunk_work_off[chunk + 1] - pl->chunk_work_off[chunk]);
    const size_t sms = (size_t)(max_blocks > 0 && max_blocks < pl->num_sms ? max_blocks : pl->num_sms);
    if (chunk < 0 && sms < (size_t)pl->num_sms && n > (size_t)pl->num_sms) return 0;
    return (int)(n < sms ? n : sms);
}
}  // namespace tessera
