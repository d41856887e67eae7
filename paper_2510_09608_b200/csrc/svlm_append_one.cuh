// The bookkeeping of ONE appended token (every decode step), shared by the append's own kernel (svlm_meta.cu) and by the decode
// kernels that do it themselves (svlm_decode.cu): what the token changes, from the control block alone, and the change.
#pragma once
#include <cuda_runtime.h>
#include "svlm_dev.h"

struct SvlmOneToken {
    long long gid, ord, u;       // stream ordinal, ordinal of its type, ring ordinal (if it is not a sink)
    long long cursor;            // native position cursor behind it
    int a, c[3];                 // native cursor advance; contiguous position
    int ty, n_tiles0, sink_fill0, n_stored0, free_top0;
    int at;                      // of the page list: the entry that grows, or where one appears
    int sink_slot;               // a sink's slot
    bool ok, is_sink, adds, new_page;      // ok: it fits; adds: an entry appears; new_page: its page comes from the free stack
};

// What the rule of a cache needs of its configuration (frozen by the first append).
struct SvlmOneRule {
    int n_sink, sink_any, contiguous, capacity, sink_slots;
    __device__ __forceinline__ explicit SvlmOneRule(const SvlmCacheDev& cd)
        : n_sink(cd.n_sink), sink_any(cd.sink_any), contiguous(cd.contiguous), capacity(cd.capacity), sink_slots(cd.n_sink_pages * SVLM_PAGE) {}
};

// The list is: sink pages, text ring pages, vision ring pages.  One token changes one entry (the last page of its ring, or
// of the sinks, grows by one slot) or adds one (a page opens), which shifts the entries behind it.
__device__ __forceinline__ SvlmOneToken svlm_one_token(const SvlmOneRule& cd, const SvlmCtrl& c, int ty, const int (&p)[3]) {
    SvlmOneToken t;
    t.ty = ty;
    t.gid = c.n_total;
    t.ord = ty ? c.n_type[1] : c.n_type[0];        // (no indexing: the arrays stay in registers)
    t.u = ty ? c.ring_n[1] : c.ring_n[0];
    t.n_tiles0 = c.n_tiles; t.sink_fill0 = c.sink_fill; t.n_stored0 = c.n_stored; t.free_top0 = c.free_top;
    t.is_sink = cd.sink_any ? t.gid < cd.n_sink : ty == 0 && t.ord < cd.n_sink;
    t.sink_slot = (int)(cd.sink_any ? t.gid : t.ord);
    t.new_page = !t.is_sink && t.u % SVLM_PAGE == 0;
    const int ns0 = (t.sink_fill0 + SVLM_PAGE - 1) / SVLM_PAGE;
    int cnt0[2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
        cnt0[k] = c.ring_n[k] > c.ring_lo[k] ? (int)((c.ring_n[k] - 1) / SVLM_PAGE - c.ring_lo[k] / SVLM_PAGE + 1) : 0;
    if (t.is_sink) {
        t.adds = t.sink_fill0 % SVLM_PAGE == 0;
        t.at = t.adds ? ns0 : ns0 - 1;
    } else {
        const long long lo = ty ? c.ring_lo[1] : c.ring_lo[0];
        const int had = ty ? cnt0[1] : cnt0[0];
        t.adds = (int)(t.u / SVLM_PAGE - lo / SVLM_PAGE + 1) != had;
        t.at = ns0 + (ty ? cnt0[0] : 0) + (t.adds ? had : had - 1);
    }
    t.ok = t.n_stored0 + 1 <= cd.capacity && (!t.new_page || t.free_top0 >= 1) && (!t.is_sink || t.sink_fill0 + 1 <= cd.sink_slots);
    const long long top = (long long)max(p[0], max(p[1], p[2])) + 1, shift = cd.contiguous ? c.shift_total : 0;
    t.a = (int)max(0ll, top - c.cursor);
    t.cursor = max(c.cursor, top);
    for (int k = 0; k < 3; ++k) t.c[k] = (int)(p[k] - shift);
    return t;
}

// Its slot.  (Where no entry appears the page could be taken from the list as well, which some callers have at hand.)
__device__ __forceinline__ int svlm_one_slot(const SvlmCacheDev& cd, const SvlmOneToken& t) {
    if (t.is_sink) return t.sink_slot;
    const int page = t.new_page ? cd.free_stack[t.free_top0 - 1] : cd.page_table[t.ty][(int)(t.u / SVLM_PAGE) & (cd.pt_size - 1)];
    return page * SVLM_PAGE + (int)(t.u % SVLM_PAGE);
}

// By one thread: everything but the shift of the list's entries behind a new one.
__device__ __forceinline__ void svlm_one_commit(const SvlmCacheDev& cd, const SvlmOneToken& t, int slot) {
    SvlmCtrl* ctrl = cd.ctrl;
    if (!t.ok) {
        ctrl->append_n = 0;
        if (ctrl->status == 0) ctrl->status = -2;   // SVLM_ERR_CAPACITY
        return;
    }
    if (t.new_page) {
        cd.page_table[t.ty][(int)(t.u / SVLM_PAGE) & (cd.pt_size - 1)] = slot / SVLM_PAGE;
        ctrl->free_top = t.free_top0 - 1;
    }
    SvlmTile* tile = cd.tiles + t.at;
    if (t.adds) {
        SvlmTile tl;
        tl.page = slot / SVLM_PAGE;
        tl.lo = slot % SVLM_PAGE;
        tl.hi = tl.lo + 1;
        tl.pad = 0;
        tl.min_gid = tl.max_gid = t.gid;
        *tile = tl;
        ctrl->n_tiles = t.n_tiles0 + 1;
    } else {
        tile->hi = slot % SVLM_PAGE + 1;
        tile->max_gid = t.gid;
    }
    cd.slot_gid[slot] = t.gid;
    cd.slot_type[slot] = (unsigned char)t.ty;
    cd.slot_a[slot] = t.a;
    cd.slot_delta[slot] = 0;
    cd.new_slot[0] = slot;
    for (int k = 0; k < 3; ++k) cd.slot_c[k * cd.n_slots + slot] = t.c[k];
    ctrl->n_total = t.gid + 1;
    ctrl->n_type[t.ty] = t.ord + 1;
    ctrl->cursor = t.cursor;
    if (t.is_sink) {
        ctrl->sink_cnt[t.ty] += 1;
        ctrl->sink_fill = t.sink_fill0 + 1;
    } else {
        ctrl->ring_n[t.ty] = t.u + 1;
    }
    ctrl->n_stored = t.n_stored0 + 1;
    ctrl->append_n = 1;
}
