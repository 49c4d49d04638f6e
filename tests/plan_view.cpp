// What the host's planner hands to the attention kernel, for tests on the CPU.  Linked with the library's host sources
// and fake_cuda.cpp.
#include <cstring>

#include "plan.h"

extern "C" {
// Copies the work list (which = 0) or the list by request chunks (1), 12 integers an item; returns its length.
__attribute__((visibility("default"))) int view_work(const tessera_plan *p, int which, int32_t *out, int room) {
    const auto &list = which ? p->work_chunked : p->work;
    if ((int)list.size() <= room) memcpy(out, list.data(), list.size() * sizeof(list[0]));
    return (int)list.size();
}
// Steps of 128 keys of every tile.
__attribute__((visibility("default"))) int view_tile_steps(const tessera_plan *p, int32_t *out, int room) {
    for (int i = 0; i < (int)p->tiles.size() && i < room; ++i) out[i] = (p->tiles[i].kv_len + 127) / 128;
    return (int)p->tiles.size();
}
__attribute__((visibility("default"))) int view_grid(const tessera_plan *p, int chunk, int max_blocks) { return tessera::attn_grid(p, chunk, max_blocks); }
__attribute__((visibility("default"))) int view_chunks(const tessera_plan *p) { return (int)p->chunk_work_off.size() - 1; }
}
