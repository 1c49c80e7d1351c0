// The test's side of fake_cuda.cpp that knows the library's handles: fields of a
// sketch, and the counters that a sampling pass's kernels would have left.
#include <string>
#include <vector>

#include "skis_internal.cuh"

namespace {
struct Pass {
    uint64_t novf, arena, n_big;
};
skis_sketch* g_sketch = nullptr;  // the sketch whose sampling passes are scripted
std::vector<Pass> g_passes;
size_t g_next = 0;
}  // namespace

extern "C" {

uint64_t fk_live(const void* p);

// counters of the next sampling passes of sketch s: n triples (novf, arena entries reserved, n_big)
void fk_script(skis_sketch* s, const uint64_t* v, int n) {
    g_sketch = s;
    g_passes.clear();
    g_next = 0;
    for (int i = 0; i < n; ++i) g_passes.push_back({v[3 * i], v[3 * i + 1], v[3 * i + 2]});
}

void fk_on_launch(const char* kernel) {
    const std::string name(kernel);
    if (name.find("k_iis_warp") == std::string::npos && name.find("k_lt_mid") == std::string::npos) return;
    if (!g_sketch || g_next >= g_passes.size()) return;  // the second tier is launched once a pass
    const Pass& p = g_passes[g_next++];
    g_sketch->ctr->novf = p.novf;
    g_sketch->ctr->arena += p.arena;
    if (g_sketch->ctr->arena > g_sketch->arena_cap && !p.novf) g_sketch->ctr->novf = 1;  // the last one does not fit
    g_sketch->ctr->n_big = p.n_big;
}

// the graph's sum of w (no kernel ran that would have computed it)
void fk_set_W(skis_graph* g, uint64_t W) { g->W = W; }
// a plain field of the sketch
uint64_t fk_value(const skis_sketch* s, const char* f) {
    const std::string n(f);
#define FIELD(x) \
    if (n == #x) return (uint64_t)s->x;
    FIELD(T) FIELD(hcap) FIELD(list_cap) FIELD(arena_cap) FIELD(spill_warps) FIELD(cta_slots_alloc) FIELD(queue_cap)
    FIELD(bitmap_words) FIELD(big_slots) FIELD(lean) FIELD(lt_mid_lanes) FIELD(smask_cap) FIELD(touched_cap)
#undef FIELD
    return ~0ull;
}
// live bytes behind a pointer of the sketch (0: null or freed)
uint64_t fk_bytes(const skis_sketch* s, const char* f) {
    const std::string n(f);
    const void* p = nullptr;
#define FIELD(x) \
    if (n == #x) p = s->x;
    FIELD(h_off) FIELD(h_len) FIELD(h_src) FIELD(h_retries) FIELD(h_coins) FIELD(arena) FIELD(ctr) FIELD(status)
    FIELD(to_warp_ids) FIELD(to_cta_ids) FIELD(ovf_ids[0]) FIELD(ovf_ids[1]) FIELD(srcrec) FIELD(srcpick)
    FIELD(spill_hash) FIELD(spill_queue) FIELD(bitmaps) FIELD(slot_clean) FIELD(queues) FIELD(big_ids) FIELD(big_queues)
    FIELD(lt_hash) FIELD(lt_list) FIELD(smask) FIELD(qmask) FIELD(qbits) FIELD(qcov) FIELD(touched) FIELD(ntouched)
    FIELD(hits) FIELD(qstatus)
#undef FIELD
    return fk_live(p);
}
uint64_t fk_cursor(const skis_sketch* s) { return s->ctr ? s->ctr->arena : 0; }
uint64_t fk_first_bad(const skis_sketch* s) { return s->qstatus->first_bad; }
int fk_events(const skis_sketch* s) { return s->ev[0] && s->ev[1] && s->ev[2] && s->ev[3]; }

}  // extern "C"
