// Metadata kernels: token bookkeeping on append, and the keep-mask / prefix-scan / re-index step
// of eviction (paper Section 2.1, "Streaming-aware KV Cache" and "Contiguous RoPE").  Integer work
// only; one CTA each (a few thousand records), results must be bit-exact.
#include <cuda_runtime.h>

#include <algorithm>

#include "svlm_append_one.cuh"
#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_ptx.cuh"
#include "svlm_rotate.cuh"

namespace {

constexpr int META_THREADS = 1024;
constexpr int META_WARPS = META_THREADS / 32;

// Block-wide exclusive scans over one value per thread.  `carry` is the running value over all
// earlier rounds; on return every thread holds the exclusive result including the carry, and carry
// has been advanced by this round's total.  All threads of the block must call.
__device__ int block_excl_sum(int v, int& carry, int* warp_buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_buf[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = warp_buf[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        warp_buf[lane] = w;   // inclusive over warps
    }
    __syncthreads();
    const int before = (warp ? warp_buf[warp - 1] : 0);
    const int total = warp_buf[META_WARPS - 1];
    const int res = carry + before + inc - v;
    __syncthreads();
    carry += total;
    return res;
}

template <int WARPS>
__device__ long long block_excl_sum64(long long v, long long& carry, long long* warp_buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_buf[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < WARPS ? warp_buf[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        if (lane < WARPS) warp_buf[lane] = w;
    }
    __syncthreads();
    const long long before = (warp ? warp_buf[warp - 1] : 0);
    const long long total = warp_buf[WARPS - 1];
    const long long res = carry + before + inc - v;
    __syncthreads();
    carry += total;
    return res;
}

// Exclusive prefix maximum (carry = maximum over everything earlier).
__device__ long long block_excl_max64(long long v, long long& carry, long long* warp_buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long NEG = -(1ll << 62);
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = max(inc, t);
    }
    long long exc = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) exc = NEG;
    if (lane == 31) warp_buf[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        long long w = warp_buf[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w = max(w, t);
        }
        warp_buf[lane] = w;
    }
    __syncthreads();
    const long long before = (warp ? warp_buf[warp - 1] : NEG);
    const long long total = warp_buf[META_WARPS - 1];
    const long long res = max(carry, max(before, exc));
    __syncthreads();
    carry = max(carry, total);
    return res;
}

__device__ __forceinline__ int ring_slot(const SvlmCacheDev& cd, int type, long long u) {
    const int page = cd.page_table[type][(int)(u / SVLM_PAGE) & (cd.pt_size - 1)];
    return page * SVLM_PAGE + (int)(u % SVLM_PAGE);
}

__device__ __forceinline__ long long ceil_page(long long x) { return (x + SVLM_PAGE - 1) / SVLM_PAGE; }

// The list of active pages: sink pages, then the text ring, then the vision ring.
struct TileList {
    int n_sink_tiles, sink_fill, cnt[2], total;
    long long first[2], lo[2], n[2];
    __device__ __forceinline__ TileList(int sink_fill_, const long long ring_lo[2], const long long ring_n[2]) : sink_fill(sink_fill_) {
        n_sink_tiles = (sink_fill + SVLM_PAGE - 1) / SVLM_PAGE;
        for (int t = 0; t < 2; ++t) {
            lo[t] = ring_lo[t];
            n[t] = ring_n[t];
            first[t] = ring_lo[t] / SVLM_PAGE;
            cnt[t] = ring_n[t] > ring_lo[t] ? (int)((ring_n[t] - 1) / SVLM_PAGE - first[t] + 1) : 0;
        }
        total = n_sink_tiles + cnt[0] + cnt[1];
    }
    // Entry i without its ordinals; page_of(type, ring page) names the physical page.
    template <typename PageOf>
    __device__ __forceinline__ SvlmTile entry(int i, PageOf page_of) const {
        SvlmTile tl;
        if (i < n_sink_tiles) {
            tl.page = i;
            tl.lo = 0;
            tl.hi = min(SVLM_PAGE, sink_fill - i * SVLM_PAGE);
        } else {
            const int t = (i - n_sink_tiles < cnt[0]) ? 0 : 1;
            const long long k = first[t] + (i - n_sink_tiles - (t ? cnt[0] : 0));
            tl.page = page_of(t, k);
            tl.lo = (int)max(0ll, lo[t] - k * SVLM_PAGE);
            tl.hi = (int)min((long long)SVLM_PAGE, n[t] - k * SVLM_PAGE);
        }
        tl.pad = 0;
        tl.min_gid = tl.max_gid = 0;
        return tl;
    }
};

// Called by all threads after the slot metadata of this kernel has been written and synchronised.
__device__ void rebuild_tiles(const SvlmCacheDev& cd, int sink_fill, const long long ring_lo[2], const long long ring_n[2]) {
    const TileList list(sink_fill, ring_lo, ring_n);
    for (int i = threadIdx.x; i < list.total; i += blockDim.x) {
        SvlmTile tl = list.entry(i, [&](int t, long long k) { return cd.page_table[t][(int)k & (cd.pt_size - 1)]; });
        tl.min_gid = cd.slot_gid[tl.page * SVLM_PAGE + tl.lo];
        tl.max_gid = cd.slot_gid[tl.page * SVLM_PAGE + tl.hi - 1];
        cd.tiles[i] = tl;
    }
    if (threadIdx.x == 0) cd.ctrl->n_tiles = list.total;
}

// ---------------------------------------------------------------------------------------------
// Append of ONE token (every decode step): the same bookkeeping as the general kernel below without its
// block-wide scans, and with the list of active pages edited instead of rebuilt: a single token changes
// one entry (the last page of its ring, or of the sinks, grows by one slot) or adds one (a page opens),
// which shifts the entries behind it.  The old entries are fetched while the control block is still on
// its way, so the kernel is two dependent round trips (control block, then page table or free stack)
// instead of six.  A block of 128 threads with a few entries each: it finds room beside the decode step before it and is
// resident when that one ends.
constexpr int ONE_THREADS = 128;
constexpr int ONE_ENTRIES = 4;      // list entries per thread
__device__ __forceinline__ void append_one_body(const SvlmCacheDev& cd, const unsigned char* types, const int* pos) {
    const int tid = threadIdx.x;
    SvlmTile old[ONE_ENTRIES];    // entries tid, tid + 128, ... of the present list (garbage beyond its end; never used then)
#pragma unroll
    for (int k = 0; k < ONE_ENTRIES; ++k)
        if (tid + k * ONE_THREADS < cd.n_pages) old[k] = cd.tiles[tid + k * ONE_THREADS];
    const SvlmCtrl ctrl = *cd.ctrl;
    const int ty = types[0] ? 1 : 0, pw = cd.rope_mode == 0 ? 0 : 1;
    const int p[3] = {pos[0], pos[pw], pos[2 * pw]};
    const SvlmOneToken t = svlm_one_token(SvlmOneRule(cd), ctrl, ty, p);
    __syncthreads();              // every old entry is in registers
    if (t.ok && t.adds)           // entries behind the new one move up by one
#pragma unroll
        for (int k = 0; k < ONE_ENTRIES; ++k) {
            const int i = tid + k * ONE_THREADS;
            if (i < t.n_tiles0 && i >= t.at) cd.tiles[i + 1] = old[k];
        }
    if (tid == 0) svlm_one_commit(cd, t, t.ok ? svlm_one_slot(cd, t) : 0);
}

// ---------------------------------------------------------------------------------------------
// Append of up to blockDim tokens, one per thread (a chunk): the general kernel's bookkeeping in three dependent round
// trips (control block with types and positions; page table or free stack; ordinals for the page list) and two block
// barriers.  Every warp adds up all warps' totals for itself, and every thread knows which page of the free stack its
// ring page becomes, so that nothing waits for one thread's page allocation.  placed(slot, c) is called for the thread's token
// with its slot and position.  False if the append was dropped (the same in every thread).
template <typename Placed>
__device__ __forceinline__ bool append_few_body(const SvlmCacheDev& cd, const unsigned char* types, const int* pos, int n, Placed placed) {
    __shared__ int s_text[META_WARPS], s_sink[META_WARPS];       // per warp: text tokens; text tokens among the any-type sinks
    __shared__ long long s_top[META_WARPS];                      // per warp: largest native index + 1
    SvlmCtrl* ctrl = cd.ctrl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = blockDim.x >> 5;
    const long long NEG = -(1ll << 62);
    const bool live = tid < n;
    const int ty = live ? (types[tid] ? 1 : 0) : 1;
    long long p[3] = {0, 0, 0};
    if (live) {
        if (cd.rope_mode == 0) { p[0] = p[1] = p[2] = pos[tid]; }
        else { p[0] = pos[3 * tid]; p[1] = pos[3 * tid + 1]; p[2] = pos[3 * tid + 2]; }
    }
    const long long n_total0 = ctrl->n_total;
    const long long nt0[2] = {ctrl->n_type[0], ctrl->n_type[1]};
    const long long cursor0 = ctrl->cursor;
    const long long shift = cd.contiguous ? ctrl->shift_total : 0;
    const long long ring_n0[2] = {ctrl->ring_n[0], ctrl->ring_n[1]};
    const long long ring_lo0[2] = {ctrl->ring_lo[0], ctrl->ring_lo[1]};
    const int sink_cnt0[2] = {ctrl->sink_cnt[0], ctrl->sink_cnt[1]};
    const int sink_fill0 = ctrl->sink_fill;
    const int n_stored0 = ctrl->n_stored;
    const int free_top0 = ctrl->free_top;

    // inside the warp
    const long long any_limit = (long long)cd.n_sink - n_total0;   // tokens i < any_limit are sinks (any-type policy)
    const unsigned text_mask = __ballot_sync(0xffffffffu, live && ty == 0);
    const unsigned sink_mask = __ballot_sync(0xffffffffu, live && ty == 0 && cd.sink_any && tid < any_limit);
    const long long top = live ? max(p[0], max(p[1], p[2])) + 1 : NEG;
    long long inc = top;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = max(inc, t);
    }
    long long exc = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) exc = NEG;
    if (lane == 31) { s_text[warp] = __popc(text_mask); s_sink[warp] = __popc(sink_mask); s_top[warp] = inc; }
    __syncthreads();
    // over the warps, by every warp
    int w_text = lane < n_warps ? s_text[lane] : 0, w_sink = lane < n_warps ? s_sink[lane] : 0;
    long long w_top = lane < n_warps ? s_top[lane] : NEG;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, w_text, o), k = __shfl_up_sync(0xffffffffu, w_sink, o);
        const long long m = __shfl_up_sync(0xffffffffu, w_top, o);
        if (lane >= o) { w_text += t; w_sink += k; w_top = max(w_top, m); }
    }
    const int n_text_new = __shfl_sync(0xffffffffu, w_text, 31), n_sink_text = __shfl_sync(0xffffffffu, w_sink, 31);
    const long long top_all = __shfl_sync(0xffffffffu, w_top, 31);
    const int text_earlier = __shfl_sync(0xffffffffu, w_text, max(warp - 1, 0));
    const long long top_earlier = __shfl_sync(0xffffffffu, w_top, max(warp - 1, 0));
    const int text_before = (warp ? text_earlier : 0) + __popc(text_mask & ((1u << lane) - 1));
    const long long cur_before = max(cursor0, max(warp ? top_earlier : NEG, exc));

    // totals, the same in every thread
    int sink_new[2];
    if (cd.sink_any) {
        const int sinks = (int)max(0ll, min(any_limit, (long long)n));
        sink_new[0] = n_sink_text;
        sink_new[1] = sinks - n_sink_text;
    } else {   // the first n_sink text ordinals are the sinks
        sink_new[0] = (int)max(0ll, min((long long)cd.n_sink - nt0[0], (long long)n_text_new));
        sink_new[1] = 0;
    }
    const int new_by_type[2] = {n_text_new, n - n_text_new};
    long long ring_n1[2], open0[2];       // open0: first ring page this append opens
    int opened[2];
    for (int t = 0; t < 2; ++t) {
        ring_n1[t] = ring_n0[t] + new_by_type[t] - sink_new[t];
        open0[t] = ceil_page(ring_n0[t]);
        opened[t] = (int)(ceil_page(ring_n1[t]) - open0[t]);
    }
    const int sink_fill1 = sink_fill0 + sink_new[0] + sink_new[1];
    if (n_stored0 + n > cd.capacity || opened[0] + opened[1] > free_top0 || sink_fill1 > cd.n_sink_pages * SVLM_PAGE) {
        if (tid == 0) {
            ctrl->append_n = 0;
            if (ctrl->status == 0) ctrl->status = -2;   // SVLM_ERR_CAPACITY
        }
        return false;
    }
    // ring page k of type t: an open one from the page table, a new one from the free stack (text ring's first)
    auto page_of = [&](int t, long long k) {
        return k < open0[t] ? cd.page_table[t][(int)k & (cd.pt_size - 1)] : cd.free_stack[free_top0 - 1 - (int)(k - open0[t]) - (t ? opened[0] : 0)];
    };
    for (int i = tid; i < opened[0] + opened[1]; i += blockDim.x) {
        const int t = i < opened[0] ? 0 : 1;
        cd.page_table[t][(int)(open0[t] + (t ? i - opened[0] : i)) & (cd.pt_size - 1)] = cd.free_stack[free_top0 - 1 - i];
    }
    if (live) {
        const long long gid = n_total0 + tid;
        const long long ord = nt0[ty] + (ty == 0 ? text_before : tid - text_before);
        const bool is_sink = cd.sink_any ? (gid < cd.n_sink) : (ty == 0 && ord < cd.n_sink);
        int slot;
        if (is_sink) {
            slot = (int)(cd.sink_any ? gid : ord);
        } else {
            const long long u = ord - (sink_cnt0[ty] + sink_new[ty]);
            slot = page_of(ty, u / SVLM_PAGE) * SVLM_PAGE + (int)(u % SVLM_PAGE);
        }
        cd.slot_gid[slot] = gid;
        cd.slot_type[slot] = (unsigned char)ty;
        cd.slot_a[slot] = (int)max(0ll, top - cur_before);
        cd.slot_delta[slot] = 0;
        cd.new_slot[tid] = slot;
        const int c[3] = {(int)(p[0] - shift), (int)(p[1] - shift), (int)(p[2] - shift)};
        for (int k = 0; k < 3; ++k) cd.slot_c[k * cd.n_slots + slot] = c[k];
        placed(slot, c);
    }
    // the list of active pages: which page and which offsets are known already, the ordinals behind the barrier
    const TileList tl(sink_fill1, ring_lo0, ring_n1);
    SvlmTile mine;
    if (tid < tl.total) mine = tl.entry(tid, page_of);
    __syncthreads();                      // the new tokens' ordinals are in place
    for (int i = tid; i < tl.total; i += blockDim.x) {
        if (i != tid) mine = tl.entry(i, page_of);
        mine.min_gid = cd.slot_gid[mine.page * SVLM_PAGE + mine.lo];
        mine.max_gid = cd.slot_gid[mine.page * SVLM_PAGE + mine.hi - 1];
        cd.tiles[i] = mine;
    }
    if (tid == 0) {
        ctrl->n_tiles = tl.total;
        ctrl->free_top = free_top0 - opened[0] - opened[1];
        ctrl->n_total = n_total0 + n;
        ctrl->n_type[0] = nt0[0] + new_by_type[0];
        ctrl->n_type[1] = nt0[1] + new_by_type[1];
        ctrl->cursor = max(cursor0, top_all);
        ctrl->ring_n[0] = ring_n1[0];
        ctrl->ring_n[1] = ring_n1[1];
        ctrl->sink_cnt[0] = sink_cnt0[0] + sink_new[0];
        ctrl->sink_cnt[1] = sink_cnt0[1] + sink_new[1];
        ctrl->sink_fill = sink_fill1;
        ctrl->n_stored = n_stored0 + n;
        ctrl->append_n = n;
    }
    return true;
}

// ---------------------------------------------------------------------------------------------
// Append: stream ordinal, per-type ordinal, cursor advance a = max(0, max(p)+1 - cursor),
// contiguous position c = p - shift_total, and the storage slot of each of the n new tokens.
__device__ __forceinline__ void append_meta_body(const SvlmCacheDev& cd, const unsigned char* types, const int* pos,
                                                 int n) {
    __shared__ int wbuf[META_WARPS];
    __shared__ long long wbuf64[META_WARPS];
    __shared__ int s_cnt[3];     // text tokens; sink tokens of type TEXT / VISION in this append
    __shared__ int s_ok;
    SvlmCtrl* ctrl = cd.ctrl;
    const int tid = threadIdx.x;
    if (tid < 3) s_cnt[tid] = 0;
    __syncthreads();

    const long long n_total0 = ctrl->n_total;
    const long long nt0[2] = {ctrl->n_type[0], ctrl->n_type[1]};
    const long long cursor0 = ctrl->cursor;
    const long long shift = cd.contiguous ? ctrl->shift_total : 0;
    const long long ring_n0[2] = {ctrl->ring_n[0], ctrl->ring_n[1]};
    const long long ring_lo0[2] = {ctrl->ring_lo[0], ctrl->ring_lo[1]};
    const int sink_cnt0[2] = {ctrl->sink_cnt[0], ctrl->sink_cnt[1]};
    const int sink_fill0 = ctrl->sink_fill;
    const int n_stored0 = ctrl->n_stored;
    const int free_top0 = ctrl->free_top;

    // pass 0: totals
    {
        int text = 0, sink_text = 0, sink_vis = 0;
        const long long any_limit = (long long)cd.n_sink - n_total0;   // tokens i < any_limit are sinks (any-type policy)
        for (int i = tid; i < n; i += META_THREADS) {
            const int ty = types[i] ? 1 : 0;
            text += (ty == 0);
            if (cd.sink_any && i < any_limit) { sink_text += (ty == 0); sink_vis += (ty == 1); }
        }
        atomicAdd(&s_cnt[0], text);
        atomicAdd(&s_cnt[1], sink_text);
        atomicAdd(&s_cnt[2], sink_vis);
    }
    __syncthreads();
    const int n_text_new = s_cnt[0];
    int sink_new[2];
    if (cd.sink_any) {
        sink_new[0] = s_cnt[1];
        sink_new[1] = s_cnt[2];
    } else {   // the first n_sink text ordinals are the sinks
        long long room = (long long)cd.n_sink - nt0[0];
        sink_new[0] = (int)max(0ll, min(room, (long long)n_text_new));
        sink_new[1] = 0;
    }
    const int new_by_type[2] = {n_text_new, n - n_text_new};
    long long ring_n1[2];
    int pages_needed = 0;
    for (int t = 0; t < 2; ++t) {
        ring_n1[t] = ring_n0[t] + new_by_type[t] - sink_new[t];
        pages_needed += (int)(ceil_page(ring_n1[t]) - ceil_page(ring_n0[t]));
    }
    if (tid == 0) {
        const bool ok = (n_stored0 + n <= cd.capacity) && (pages_needed <= free_top0) &&
                        (sink_fill0 + sink_new[0] + sink_new[1] <= cd.n_sink_pages * SVLM_PAGE);
        s_ok = ok;
        if (!ok) {
            ctrl->append_n = 0;
            if (ctrl->status == 0) ctrl->status = -2;   // SVLM_ERR_CAPACITY
        } else {   // take pages for the ring ordinals this append opens
            int top = free_top0;
            for (int t = 0; t < 2; ++t)
                for (long long k = ceil_page(ring_n0[t]); k < ceil_page(ring_n1[t]); ++k)
                    cd.page_table[t][(int)k & (cd.pt_size - 1)] = cd.free_stack[--top];
            ctrl->free_top = top;
        }
    }
    __syncthreads();
    if (!s_ok) return;

    // pass 1: per-token scans, in rounds of one token per thread
    int text_carry = 0;
    long long top_carry = cursor0;
    const int sink_final[2] = {sink_cnt0[0] + sink_new[0], sink_cnt0[1] + sink_new[1]};
    for (int base = 0; base < n; base += META_THREADS) {
        const int i = base + tid;
        const bool live = i < n;
        const int ty = live ? (types[i] ? 1 : 0) : 1;
        long long p[3] = {0, 0, 0};
        if (live) {
            if (cd.rope_mode == 0) { p[0] = p[1] = p[2] = pos[i]; }
            else { p[0] = pos[3 * i]; p[1] = pos[3 * i + 1]; p[2] = pos[3 * i + 2]; }
        }
        const long long top = live ? max(p[0], max(p[1], p[2])) + 1 : -(1ll << 62);
        const int text_before = block_excl_sum(live && ty == 0, text_carry, wbuf);
        const long long cur_before = block_excl_max64(top, top_carry, wbuf64);
        if (!live) continue;
        const long long gid = n_total0 + i;
        const long long ord = nt0[ty] + (ty == 0 ? text_before : i - text_before);
        const long long a = max(0ll, top - cur_before);
        const bool is_sink = cd.sink_any ? (gid < cd.n_sink) : (ty == 0 && ord < cd.n_sink);
        int slot;
        if (is_sink) slot = (int)(cd.sink_any ? gid : ord);
        else slot = ring_slot(cd, ty, ord - sink_final[ty]);
        cd.slot_gid[slot] = gid;
        cd.slot_type[slot] = (unsigned char)ty;
        cd.slot_a[slot] = (int)a;
        cd.slot_delta[slot] = 0;
        cd.new_slot[i] = slot;
        for (int k = 0; k < 3; ++k) cd.slot_c[k * cd.n_slots + slot] = (int)(p[k] - shift);
    }
    __syncthreads();
    const int sink_fill1 = sink_fill0 + sink_new[0] + sink_new[1];
    rebuild_tiles(cd, sink_fill1, ring_lo0, ring_n1);
    if (tid == 0) {
        ctrl->n_total = n_total0 + n;
        ctrl->n_type[0] = nt0[0] + new_by_type[0];
        ctrl->n_type[1] = nt0[1] + new_by_type[1];
        ctrl->cursor = top_carry;
        ctrl->ring_n[0] = ring_n1[0];
        ctrl->ring_n[1] = ring_n1[1];
        ctrl->sink_cnt[0] = sink_final[0];
        ctrl->sink_cnt[1] = sink_final[1];
        ctrl->sink_fill = sink_fill1;
        ctrl->n_stored = n_stored0 + n;
        ctrl->append_n = n;
    }
}

// Number of entries of the sorted list g[0..n) that are smaller than key.
__device__ __forceinline__ int count_below(const long long* g, int n, long long key) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (g[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

constexpr int ROTATE_THREADS = 256;
constexpr int EV_SMEM = 2048;   // evicted tokens of one call whose lists also fit in shared memory
constexpr int KEPT_BATCH = 2;   // retained tokens a thread handles per round (loads of a round are issued together)
constexpr int EV_CLUSTER = 8;   // most CTAs (one thread-block cluster) that share the retained tokens of one cache
constexpr int EV_PER_CTA = KEPT_BATCH * META_THREADS;   // retained tokens of a CTA and round
// A cluster just large enough for one round (a small cache needs no cluster barrier across CTAs at all).
int evict_cluster(int capacity) {
    int c = 1;
    while (c < EV_CLUSTER && c * EV_PER_CTA < capacity) c *= 2;
    return c;
}

__device__ __forceinline__ unsigned cluster_ctarank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_nctarank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// All threads of all CTAs of the cluster; orders their global-memory accesses before the arrival and after the wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// Evict: keep-mask (a suffix of each ring plus the sinks), prefix sums of the evicted tokens'
// cursor advances, and the left-shift E(i) of every retained token i: the advances of all evicted
// tokens that precede it in the stream.
//
// The kernel is a chain of dependent round trips to L2 (control block -> page table -> ordinals, advances, positions ->
// search -> stores), so a round's loads are all issued together: the retained tokens', the evicted tokens' and the page
// list's.  A cluster of CTAs serves one cache: every CTA builds the (short) evicted lists for itself, the retained tokens
// are dealt out among the CTAs, the last CTA writes the page list, and CTA 0 alone changes what the others read (behind
// the cluster barrier) and keeps the books.  The chain had ten round trips, one stage after another: 11.9 us at config 3,
// 7 now (append and eviction of a chunk in a row: 22.6 -> 17.4 us).
//
// ROTATE: a single CTA serves the cache (a retained token per thread at most) and re-rotates the moved keys as well, where
// that is so little that a launch of its own costs more (svlm_evict_in_one); of no more threads than that takes, since the
// barriers cost by the warp (ROTATE_THREADS).
template <bool ROTATE, int THREADS>
__device__ __forceinline__ void evict_meta_body(const SvlmCacheDev& cd) {
    constexpr int PER_CTA = KEPT_BATCH * THREADS;           // retained tokens of a CTA and round
    const int crank = (int)cluster_ctarank(), n_ctas = (int)cluster_nctarank();
    __shared__ long long wbuf64[2][(THREADS / 32)];
    __shared__ long long s_gid[EV_SMEM];       // ordinals of the evicted tokens: text ring, then vision ring
    __shared__ long long s_pref[EV_SMEM + 2];  // exclusive prefix sums of their advances (n+1 entries per ring)
    __shared__ int s_moved;
    __shared__ int2 moved_slots[ROTATE ? THREADS : 1]; // slot and shift of the retained tokens (slot -1: none, or not moved)
    SvlmCtrl* ctrl = cd.ctrl;
    const int tid = threadIdx.x;
    if (tid == 0) s_moved = 0;

    const long long ring_n[2] = {ctrl->ring_n[0], ctrl->ring_n[1]};
    const long long lo0[2] = {ctrl->ring_lo[0], ctrl->ring_lo[1]};
    const int sink_fill = ctrl->sink_fill;
    const int free_top0 = ctrl->free_top;
    const int win[2] = {cd.text_window, cd.vision_window};
    long long lo1[2];
    int n_ev[2];
    for (int t = 0; t < 2; ++t) {
        lo1[t] = min(ring_n[t], max(lo0[t], ring_n[t] - (long long)win[t]));
        n_ev[t] = (int)(lo1[t] - lo0[t]);
    }
    const bool in_smem = n_ev[0] + n_ev[1] <= EV_SMEM;
    // where the searches read the lists of ring t
    const long long* gid_list[2] = {in_smem ? s_gid : cd.ev_gid[0], in_smem ? s_gid + n_ev[0] : cd.ev_gid[1]};
    const long long* pref_list[2] = {in_smem ? s_pref : cd.ev_pref[0], in_smem ? s_pref + n_ev[0] + 1 : cd.ev_pref[1]};

    // retained tokens: sinks, then the kept suffix of each ring; CTA r takes every n_ctas-th block of them
    const long long kept_ring[2] = {ring_n[0] - lo1[0], ring_n[1] - lo1[1]};
    const long long n_kept = sink_fill + kept_ring[0] + kept_ring[1];
    int k_slot[KEPT_BATCH], k_c[KEPT_BATCH][3];
    long long k_g[KEPT_BATCH];
    auto kept_slots = [&](long long base) {
#pragma unroll
        for (int u = 0; u < KEPT_BATCH; ++u) {
            const long long i = base + (long long)u * THREADS + tid;
            if (i >= n_kept) k_slot[u] = -1;
            else if (i < sink_fill) k_slot[u] = (int)i;
            else if (i < sink_fill + kept_ring[0]) k_slot[u] = ring_slot(cd, 0, lo1[0] + (i - sink_fill));
            else k_slot[u] = ring_slot(cd, 1, lo1[1] + (i - sink_fill - kept_ring[0]));
        }
    };
    auto kept_data = [&] {
#pragma unroll
        for (int u = 0; u < KEPT_BATCH; ++u) {
            k_g[u] = k_slot[u] >= 0 ? cd.slot_gid[k_slot[u]] : 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) k_c[u][k] = k_slot[u] >= 0 ? cd.slot_c[k * cd.n_slots + k_slot[u]] : 0;
        }
    };
    // evicted tokens of both rings, one of each per thread and round
    int e_slot[2];
    long long e_a[2], e_g[2];
    auto evicted_slots = [&](int base) {
#pragma unroll
        for (int t = 0; t < 2; ++t) e_slot[t] = base + tid < n_ev[t] ? ring_slot(cd, t, lo0[t] + base + tid) : -1;
    };
    auto evicted_data = [&] {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            e_a[t] = e_slot[t] >= 0 && cd.contiguous ? cd.slot_a[e_slot[t]] : 0;
            e_g[t] = e_slot[t] >= 0 ? cd.slot_gid[e_slot[t]] : 0;
        }
    };
    const long long base0 = (long long)crank * PER_CTA;
    const bool lists = crank == n_ctas - 1;       // this CTA writes the page list
    auto page_of = [&](int t, long long k) { return cd.page_table[t][(int)k & (cd.pt_size - 1)]; };
    evicted_slots(0);
    kept_slots(base0);
    evicted_data();
    kept_data();

    // evicted tokens in ordinal (= stream) order, with exclusive prefix sums of a
    long long freed[2] = {0, 0};
    for (int base = 0; base < max(n_ev[0], n_ev[1]); base += THREADS) {
        const int i = base + tid;
        if (base) { evicted_slots(base); evicted_data(); }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            if (base >= n_ev[t]) continue;            // uniform over the block
            const long long ex = block_excl_sum64<THREADS / 32>(e_a[t], freed[t], wbuf64[t]);
            if (e_slot[t] >= 0) {
                if (in_smem) {
                    s_gid[(t ? n_ev[0] : 0) + i] = e_g[t];
                    s_pref[(t ? n_ev[0] + 1 : 0) + i] = ex;
                } else {   // every CTA writes the same values
                    cd.ev_gid[t][i] = e_g[t];
                    cd.ev_pref[t][i] = ex;
                }
            }
        }
    }
    if (tid == 0)
        for (int t = 0; t < 2; ++t) {
            if (in_smem) s_pref[(t ? n_ev[0] + 1 : 0) + n_ev[t]] = freed[t];
            else cd.ev_pref[t][n_ev[t]] = freed[t];
        }
    if (n_ctas > 1 && crank == 0 && tid == 0) ctrl->evict_moved = 0;      // before the others' say
    __syncthreads();
    cluster_arrive();    // this CTA has read the control block and the evicted slots' metadata

    int moved = 0;
    if (ROTATE) moved_slots[tid] = make_int2(-1, 0);
    for (long long base = base0; base < n_kept; base += (long long)n_ctas * PER_CTA) {
        if (base != base0) { kept_slots(base); kept_data(); }
        int E[KEPT_BATCH];
#pragma unroll
        for (int u = 0; u < KEPT_BATCH; ++u) {
            long long e = 0;
            if (k_slot[u] >= 0)
                for (int t = 0; t < 2; ++t)
                    if (n_ev[t]) e += pref_list[t][count_below(gid_list[t], n_ev[t], k_g[u])];
            E[u] = (int)e;
        }
#pragma unroll
        for (int u = 0; u < KEPT_BATCH; ++u) {
            if (k_slot[u] < 0) continue;
            cd.slot_delta[k_slot[u]] = E[u];
            if (E[u]) {
                moved = 1;
                if (ROTATE && u == 0) moved_slots[tid] = make_int2(k_slot[u], E[u]);
#pragma unroll
                for (int k = 0; k < 3; ++k) cd.slot_c[k * cd.n_slots + k_slot[u]] = k_c[u][k] - E[u];
            }
        }
    }
    if (moved) s_moved = 1;
    const TileList tl(sink_fill, lo1, ring_n);
    if (lists)
        for (int i = tid; i < tl.total; i += THREADS) {      // (the ordinals of retained tokens do not change here)
            SvlmTile tile = tl.entry(i, page_of);
            tile.min_gid = cd.slot_gid[tile.page * SVLM_PAGE + tile.lo];
            tile.max_gid = cd.slot_gid[tile.page * SVLM_PAGE + tile.hi - 1];
            cd.tiles[i] = tile;
        }
    // release the pages that fell wholly below the new low-water mark (text ring's first, in ring order)
    long long first[2], cnt[2];
    for (int t = 0; t < 2; ++t) {
        first[t] = lo0[t] / SVLM_PAGE;
        cnt[t] = max(0ll, min(lo1[t] / SVLM_PAGE, ceil_page(ring_n[t])) - first[t]);
    }
    if (crank == 0)
        for (long long i = tid; i < cnt[0] + cnt[1]; i += THREADS) {
            const int t = i < cnt[0] ? 0 : 1;
            cd.free_stack[free_top0 + i] = page_of(t, first[t] + (t ? i - cnt[0] : i));
        }
    __syncthreads();
    cluster_wait();      // every CTA has read them: now the evicted slots can be marked empty
    if (crank == 0) {
        for (int base = 0; base < max(n_ev[0], n_ev[1]); base += THREADS) {
            if (max(n_ev[0], n_ev[1]) > THREADS) evicted_slots(base);      // (else this thread's are still at hand)
#pragma unroll
            for (int t = 0; t < 2; ++t)
                if (e_slot[t] >= 0) {
                    cd.slot_gid[e_slot[t]] = -1;
                    cd.slot_delta[e_slot[t]] = 0;
                }
        }
        if (tid == 0) {
            ctrl->n_tiles = tl.total;
            ctrl->free_top = free_top0 + (int)(cnt[0] + cnt[1]);
            ctrl->ring_lo[0] = lo1[0];
            ctrl->ring_lo[1] = lo1[1];
            ctrl->shift_total += freed[0] + freed[1];
            ctrl->n_stored = (int)n_kept;
        }
    }
    // whether any retained token moved: exactly when an evicted token with an advance precedes one, which every CTA
    // finds out for its own tokens
    if (tid == 0) {
        if (n_ctas == 1) ctrl->evict_moved = s_moved;
        else if (s_moved) atomicOr(&ctrl->evict_moved, 1);
    }
    if (ROTATE && s_moved) {                       // (moved_slots was complete at the barrier above)
        const int half = cd.head_dim / 2, gshift = cd.head_dim == 128 ? 3 : 2, rows = cd.layers * cd.kv_heads;
        const size_t stride = (size_t)cd.n_slots * cd.head_dim;
        for (int i = tid; i < (int)n_kept << gshift; i += THREADS) {
            const int2 mv = moved_slots[i >> gshift];
            if (mv.x < 0) continue;
            const int g = i & ((1 << gshift) - 1);
            uint16_t* at = cd.K + (size_t)mv.x * cd.head_dim + g * 8;
            const int c[3] = {-mv.y, -mv.y, -mv.y};      // all three indices of a token shift by the same amount
            float cs[8], sn[8];
            first_rotation(cd, g, c, cs, sn);
#pragma unroll 2
            for (int r = 0; r < rows; ++r, at += stride) {
                Bf16x8 lo = *reinterpret_cast<const Bf16x8*>(at), hi = *reinterpret_cast<const Bf16x8*>(at + half);
                rotate8(lo, hi, cs, sn);
                *reinterpret_cast<Bf16x8*>(at) = lo;
                *reinterpret_cast<Bf16x8*>(at + half) = hi;
            }
        }
    }
}

// All of these kernels are launched programmatically (svlm_launch_chained): they start while their predecessor ends, wait
// for it first and only then let their own successor start, so that whoever starts early behind them finds everything
// enqueued before them done.  Batched forms: block i serves cache i, whose descriptor it first copies from device memory
// into shared memory.  types is [n_caches][n], pos [n_caches][n] (1D) or [n_caches][n][3].
//
// FORM 1, one token: a decode step follows, one CTA per SM with a second slot free on each for the next layer's.  Started
// beside this kernel it finds one SM half taken, puts two CTAs on another, and every later layer-step of the chain
// inherits the unevenness (6.57 -> 7.27 us each); so there the successor starts when this CTA is gone.
enum { APPEND_ONE = 1, APPEND_FEW = 2, APPEND_ANY = 3 };
template <int FORM>
__device__ __forceinline__ void append_form(const SvlmCacheDev& cd, const unsigned char* types, const int* pos, int n) {
    svlm_ptx::pdl_wait();
    if (FORM != APPEND_ONE) svlm_ptx::pdl_launch_dependents();
    if (FORM == APPEND_ONE) append_one_body(cd, types, pos);
    else if (FORM == APPEND_FEW) append_few_body(cd, types, pos, n, [](int, const int (&)[3]) {});
    else append_meta_body(cd, types, pos, n);
}

template <int FORM>
__global__ void __launch_bounds__(FORM == APPEND_ONE ? ONE_THREADS : META_THREADS) append_meta_kernel(SvlmCacheDev cd, const unsigned char* types,
                                                                                                     const int* pos, int n) {
    append_form<FORM>(cd, types, pos, n);
}

template <int FORM>
__global__ void __launch_bounds__(FORM == APPEND_ONE ? ONE_THREADS : META_THREADS) append_meta_batch_kernel(SvlmCacheList list, const unsigned char* types,
                                                                                                           const int* pos, int n) {
    __shared__ SvlmCacheDev s_cd;
    svlm_load_desc(&s_cd, list.cd[blockIdx.x]);      // (frozen by the first append: no kernel writes it)
    append_form<FORM>(s_cd, types + (size_t)blockIdx.x * n, pos + (size_t)blockIdx.x * n * (s_cd.rope_mode == 0 ? 1 : 3), n);
}

// Append of a few tokens with the write of their keys and values in one launch: the block that places the tokens also rotates
// and stores their rows, a thread per (token, 8 pairs) and row of [layer][kv head].  The rows are asked for before the
// metadata, which they have nothing to do with.
constexpr long long APPEND_WRITE_ELEMENTS = 4096;      // of the appended keys (svlm_append_in_one)
constexpr int APPEND_WRITE_THREADS = APPEND_WRITE_ELEMENTS / 16, APPEND_WRITE_TOKENS = APPEND_WRITE_ELEMENTS / 64;   // (heads have 64 dims at least)
__global__ void __launch_bounds__(APPEND_WRITE_THREADS) append_meta_write_kernel(SvlmCacheDev cd, const unsigned char* types, const int* pos, int n, const uint16_t* K,
                                                                                 const uint16_t* V, int layers) {
    __shared__ int s_slot[APPEND_WRITE_TOKENS], s_c[APPEND_WRITE_TOKENS][3];
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    const int half = cd.head_dim / 2, gshift = cd.head_dim == 128 ? 3 : 2, d = cd.head_dim, rows = layers * cd.kv_heads;
    const int tid = threadIdx.x, token = (tid >> gshift) / rows, row = (tid >> gshift) % rows, g = tid & ((1 << gshift) - 1);
    const bool writes = token < n;
    Bf16x8 lo, hi;
    uint4 vlo, vhi;
    if (writes) {
        const int l = row / cd.kv_heads, h = row - l * cd.kv_heads;
        const size_t src = (((size_t)l * n + token) * cd.kv_heads + h) * d + g * 8;
        lo = bf16x8(svlm_ptx::ld_in(reinterpret_cast<const uint4*>(K + src)));
        hi = bf16x8(svlm_ptx::ld_in(reinterpret_cast<const uint4*>(K + src + half)));
        vlo = svlm_ptx::ld_in(reinterpret_cast<const uint4*>(V + src));
        vhi = svlm_ptx::ld_in(reinterpret_cast<const uint4*>(V + src + half));
    }
    const bool ok = append_few_body(cd, types, pos, n, [&](int slot, const int (&c)[3]) {
        s_slot[tid] = slot;
        for (int k = 0; k < 3; ++k) s_c[tid][k] = c[k];
    });
    if (!ok) return;
    __syncthreads();
    if (!writes) return;
    const int c[3] = {s_c[token][0], s_c[token][1], s_c[token][2]};
    float cs[8], sn[8];
    first_rotation(cd, g, c, cs, sn);
    rotate8(lo, hi, cs, sn);
    const size_t dst = ((size_t)row * cd.n_slots + s_slot[token]) * d + g * 8;
    *reinterpret_cast<Bf16x8*>(cd.K + dst) = lo;
    *reinterpret_cast<Bf16x8*>(cd.K + dst + half) = hi;
    *reinterpret_cast<uint4*>(cd.V + dst) = vlo;
    *reinterpret_cast<uint4*>(cd.V + dst + half) = vhi;
}

template <bool ROTATE>
__global__ void __launch_bounds__(ROTATE ? ROTATE_THREADS : META_THREADS) evict_meta_kernel(SvlmCacheDev cd) {
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    evict_meta_body<ROTATE, ROTATE ? ROTATE_THREADS : META_THREADS>(cd);
}

template <bool ROTATE>
__global__ void __launch_bounds__(ROTATE ? ROTATE_THREADS : META_THREADS) evict_meta_batch_kernel(SvlmCacheList list) {
    __shared__ SvlmCacheDev s_cd;
    svlm_load_desc(&s_cd, list.cd[blockIdx.x / cluster_nctarank()]);
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    evict_meta_body<ROTATE, ROTATE ? ROTATE_THREADS : META_THREADS>(s_cd);
}

int append_form_of(int n, int n_pages) {
    if (n == 1 && n_pages <= ONE_THREADS * ONE_ENTRIES) return APPEND_ONE;      // (the list's entries wait in registers)
    return n <= META_THREADS ? APPEND_FEW : APPEND_ANY;
}
int append_threads(int form, int n) {
    return form == APPEND_ONE ? ONE_THREADS : form == APPEND_ANY ? META_THREADS : n <= 96 ? 128 : (n + 31) / 32 * 32;   // (128: the page list)
}

}  // namespace

cudaError_t svlm_launch_append_meta_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, const unsigned char* types, const int* pos, int n,
                                   cudaStream_t st) {
    const int form = append_form_of(n, geom.n_pages);
    auto* kernel = form == APPEND_ONE ? append_meta_batch_kernel<APPEND_ONE> : form == APPEND_FEW ? append_meta_batch_kernel<APPEND_FEW> : append_meta_batch_kernel<APPEND_ANY>;
    return svlm_launch_chained(kernel, dim3(list.n), dim3(append_threads(form, n)), 0, 1, st, list, types, pos, n);
}

// One launch for a whole append or eviction of a small cache.  The lines: what one block moves by itself against a second launch
// on all SMs.  Append and eviction of a chunk in a row, replayed from a graph, us: 2.4 K elements of new keys written in the
// same launch 14.3, in a second one 15.3, 4 K 15.5 and 16.3, 8 K 17.4 and 16.6, 32 K 25.2 and 17.4; 8 K elements of kept keys
// re-rotated in the same launch 15.2, in a second one 16.6, 17 K 17.5 and 17.3 (one head) or 14.9 and 15.8 (two of 128), 155 K
// 32.9 and 17.7.  (By plain calls a launch less saves the host 2 us more.)
constexpr long long EVICT_ROTATE_ELEMENTS = 16384;     // of the keys that the windows keep
// An eviction in one launch also walks over the tokens that leave, with 256 threads where the other form has 1024.  Append and
// eviction of n tokens over 190 kept, one head of 64, vision, text and both in turn, us in one launch and in two: 700 20.6,
// 19.4, 22.7 and 22.2, 20.9, 22.8; 1024 20.7, 22.6, 22.7 and 22.6, 22.7, 23.9; 1536 26.8, 26.8, 28.2 and 26.8, 28.5, 27.1; 2048 28.8, 28.8,
// 30.6 and 27.3, 28.8, 28.8; 3000 35.0, 35.5, 35.9 and 32.9, 33.0, 34.7.
constexpr long long EVICT_ROTATE_LEAVING = 1024;
static_assert(EVICT_ROTATE_ELEMENTS / 64 <= ROTATE_THREADS, "a thread per retained token (heads have 64 dims at least)");
bool svlm_append_in_one(const SvlmCacheDev& cd, int layer, int n) {
    return (long long)n * (layer < 0 ? cd.layers : 1) * cd.kv_heads * cd.head_dim <= APPEND_WRITE_ELEMENTS;
}
bool svlm_evict_in_one(const SvlmCacheDev& cd, long long stored) {
    const long long windows = (long long)cd.n_sink + cd.vision_window + cd.text_window, kept = std::min(windows, (long long)cd.n_slots);
    return stored - windows <= EVICT_ROTATE_LEAVING && kept * cd.layers * cd.kv_heads * cd.head_dim <= EVICT_ROTATE_ELEMENTS;
}

cudaError_t svlm_launch_append_in_one(const SvlmCacheDev& cd, int layer, const void* K, const void* V, const unsigned char* types, const int* pos, int n, cudaStream_t st) {
    const int layers = layer < 0 ? cd.layers : 1, items = n * layers * cd.kv_heads * (cd.head_dim / 16);
    const int threads = std::max(append_threads(APPEND_FEW, n), (items + 31) / 32 * 32);
    return svlm_launch_chained(append_meta_write_kernel, dim3(1), dim3(threads), 0, 1, st, cd, types, pos, n, static_cast<const uint16_t*>(K),
                               static_cast<const uint16_t*>(V), layers);
}

cudaError_t svlm_launch_evict_meta_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, bool rotate, cudaStream_t st) {
    int c = rotate ? 1 : evict_cluster(geom.n_slots);            // (the caches share the number of pages, not the exact capacity)
    while (c > 1 && c * list.n > 96) c /= 2;        // 16 clusters of 8 do not find room at once (a CTA fills an SM)
    return svlm_launch_chained(rotate ? evict_meta_batch_kernel<true> : evict_meta_batch_kernel<false>, dim3(c * list.n), dim3(rotate ? ROTATE_THREADS : META_THREADS), 0, c, st, list);
}

cudaError_t svlm_launch_append_meta(const SvlmCacheDev& cd, const unsigned char* types, const int* pos, int n,
                             cudaStream_t st) {
    const int form = append_form_of(n, cd.n_pages);
    auto* kernel = form == APPEND_ONE ? append_meta_kernel<APPEND_ONE> : form == APPEND_FEW ? append_meta_kernel<APPEND_FEW> : append_meta_kernel<APPEND_ANY>;
    return svlm_launch_chained(kernel, dim3(1), dim3(append_threads(form, n)), 0, 1, st, cd, types, pos, n);
}

cudaError_t svlm_launch_evict_meta(const SvlmCacheDev& cd, bool rotate, cudaStream_t st) {
    const int c = rotate ? 1 : evict_cluster(cd.capacity);
    return svlm_launch_chained(rotate ? evict_meta_kernel<true> : evict_meta_kernel<false>, dim3(c), dim3(rotate ? ROTATE_THREADS : META_THREADS), 0, c, st, cd);
}
