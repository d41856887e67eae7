// Chunk-prefill attention for sm_100a: the new chunk's queries (n_q >= 2 rows) attend over the
// retained cache plus, causally, the chunk itself (paper Section 2.1: the retained KV is reused, only
// the new second of tokens is computed).  This is the one dense contraction of the path, so it runs
// on the 5th-generation tensor cores (chunks of few rows over short windows: svlm_prefill_small.cu).
//
// Work split.  A unit is 256 packed rows (row = (token, head in the GQA group)) of one KV head of one problem
// (cache, layer): two 128-row tiles A and B that share every K/V page (with 128 rows per CTA the K/V stream out of L2
// alone took as long as the whole kernel should).  One CTA per SM walks its part of a list of work that the host has
// made from the numbers of rows and an estimate of the pages (svlm_prefill_plan.h): first whole units, round by round over
// the grid (neighbouring CTAs then stream the same pages at the same time), then its share of the last one to two rounds'
// units, dealt out evenly in pages, so that no SM idles in a last wave (120 of 148 SMs had work for one stream's chunk before, 960 CTAs were 6.5
// waves for eight streams).  A unit that is cut between CTAs is merged by those that end in it, each a share of its columns, or by the last of them,
// through un-normalised pieces (O, m, l) in the cache's scratch; nothing depends on a wait (meet_pieces).
//
// Roles (384 threads, registers moved from warpgroup 2 to the softmax with setmaxnreg):
//   warps 0-3, 4-7   softmax of tile A, B, one thread per row; also that tile's query rotation and output
//   warp 8           TMA: K and V pages (128 slots, 128-byte swizzle) into one 4-stage ring, K(0) K(1) V(0) K(2) V(1) ...; it
//                    runs ahead into the next unit while the current one ends
//   warps 9, 10      issue tcgen05.mma for tile A, B: S = Q K^T into 128 TMEM columns, O += P V with P read from
//                    TMEM (no shared-memory round trip), and say to the softmax that P V is done
//   warp 11          fetches the cache's metadata, once; then it says to the softmax that S is there
// TMEM: O of both tiles (256 columns at head_dim 128), P of both (64 each, bf16), and one buffer of 128 for S that the tiles take
// in turns: S(A,0) S(B,0) S(A,1) S(B,1) ...  A tile's scores stay there only until they are in its softmax warps' registers, then
// the other tile's come, so S(j+1) of a tile is there before its P V(j) has begun and the softmax warps go from page to page
// without a wait.  (Before, P lay over its own S, and each tile was the serial chain S -> softmax -> P V -> next S.)
// Measured on the page loop (cycles per page pair, head_dim 128, clock read in an instrumented copy; tensor time is 2048 of them, and
// the special-function unit's 2048):
//   3750 -> 3490  two issuers, each one's waits under the other one's MMAs
//   3490 -> 2700  P handed over through named barriers instead of mbarriers (450 -> 50 cycles), in two halves, so that
//                 the first half's P V runs under the second half's exponentials
//   2700 -> 3200  all exponentials on the special-function unit (softmax_page), which costs less where power is the limit
//   3240 -> 3850  one buffer for S, but waits of one lane and shuffles in warps 9-11: each such step of theirs takes 300 to 700 cycles beside
//                 the softmax warps, whose exponentials, loads, shuffles and mbarrier operations go through the same queue
//                 (softmax warps waiting on the mbarriers themselves: 3200, of which 300 each for two waits that were complete)
//   3850 -> 2750  these waits as short loops of the whole warp (mbar_wait_short); -> 2600 by giving the columns away before the
//                 maximum, and with one form of the softmax for all pages
//   softmax of a page 2200 -> 1500 cycles for a warp by itself: the whole row in registers (one pass over TMEM), packed fp32 pairs
// With P over its own S -> now (28/4 heads of 128): 531 tokens over 31,000 keys with append and eviction 241 -> 220 us, eight layers of a
// second of video in a burst 690 -> 618; at the power limit all 28 layers 2471 -> 2312, four layers of 4133 tokens 1724 -> 1599.
// Per-page bookkeeping that cost a masked page 2 us (descriptor loads, two barriers and a bisection through shared
// memory) is now a few shuffles on values that arrive while the thread waits for S.
// Every mbarrier wait is bounded: on expiry the CTA records SVLM_ERR_TIMEOUT in the caches' status words, keeps up its
// named-barrier arrivals (their number depends on the work list only, their order on one another only), drains its copies, frees its TMEM
// and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_prefill_plan.h"
#include "svlm_ptx.cuh"
#include "svlm_rope.cuh"
#include "svlm_tc.cuh"

namespace {

using namespace svlm_ptx;
using namespace svlm_tc;

constexpr int PF_THREADS = 384;
constexpr int PF_RING = 4;            // K/V page stages (3: 18 % slower, the next K arrives late; 5: no faster)
constexpr int PF_MAX_TILES = 512;
constexpr int PF_CS_BYTES = 16384;    // rotation factors of one tile's tokens (5 or more heads per KV head, all at head_dim 64 with 2 or more)
// Registers per thread after the split; 216 * 256 + 72 * 128 = 168 * 384, what the block is launched with (checked at launch).
constexpr int PF_REGS_LAUNCH = 168;

template <int D>
__host__ __device__ constexpr size_t pf_slot_bytes() { return (size_t)PF_ROWS * D * 4 + PF_ROWS * 8; }

// ---- packed fp32 pairs ---------------------------------------------------------------------------------------
typedef unsigned long long u64;
__device__ __forceinline__ u64 pk64(float a, float b) { u64 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void un64(u64 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) { u64 r; asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ u64 add2(u64 a, u64 b) { u64 r; asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ u64 mul2(u64 a, u64 b) { u64 r; asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ float max3(float a, float b, float c) { float r; asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }
__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// ---- named barriers (the hardware's, not shared memory): ids ----------------------------------------------------
constexpr int BAR_ALL = 0;     // the thread block, as __syncthreads
constexpr int BAR_WG = 1;      // + tile: the softmax warpgroup alone (128)
constexpr int BAR_P1 = 3;      // + tile: first half of P is in TMEM (128 softmax + 32 issuer)
constexpr int BAR_P2 = 5;      // + tile: second half of P (128 + 32)
constexpr int BAR_READ = 7;    // + tile: its S is in registers, the columns are free (128 + 32 issuer of the S that comes there next)
constexpr int BAR_S = 11;      // + tile: S is in TMEM; the first time, the metadata is there (128 + 32 warp 11)
constexpr int BAR_PV = 13;     // + tile: P V is done: its P may be overwritten, its accumulator touched (128 + 32 issuer)
constexpr int BAR_Q = 9;       // + tile: the tile's query rows are in shared memory, its accumulator is free (128 + 32)
constexpr int BAR_META = 15;   // the metadata is there (warps 8 to 11), once; from then on
constexpr int BAR_ASKED = 15;  // an issuer has come past its product S, the tiles in turn (32 issuer + 32 warp 11)
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// Rescale the row's accumulator when its reference maximum moves (rare).  Eight columns at a time: with the row of
// scores live there are few registers left.
__device__ __forceinline__ void rescale_o(unsigned tO, int D, float corr) {
#pragma unroll 1
    for (int q = 0; q < D; q += 8) {
        float o[8];
        tmem_ld8(tO + q, o);
        tmem_wait_ld<8>(o);
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] *= corr;
        tmem_st8(tO + q, o);
    }
}

// Divisions without a branch: once-executed code runs at the pace of its fetching, and each jump over a slow path that is not taken
// is a new fetch (some 500 cycles where nothing has been there before).
// n / G for 0 <= n < 2^31 (the plan's reciprocal).
__device__ __forceinline__ int pf_div(int n, const PfPlan& plan) { return (int)(((unsigned long long)(unsigned)n * plan.g_magic) >> plan.g_shift); }
// a / b for 0 <= a, 0 < b and a quotient below 2^20: the float quotient is off by one at most.
__device__ __forceinline__ int pf_small_div(int a, int b) {
    const int q = (int)((float)a * __frcp_rn((float)b)), r = a - q * b;
    return q + (r >= b) - (r < 0);
}

// A piece of the work list.
struct PfSeg {
    int unit;                // unit of the launch
    int a, e;                // its pages [a, e) in 1/128 of all the unit's pages
    int tail;                // index among the tail's units, -1: a whole unit of the first rounds
};

// A CTA's walk over its work list.
struct PfWalk {
    int round, pos, end;
    __device__ __forceinline__ void begin(const PfPlan& plan) {
        round = 0;
        pos = plan.x[blockIdx.x];
        end = plan.x[blockIdx.x + 1];
    }
    __device__ __forceinline__ bool more(const PfPlan& plan) const { return round < plan.rounds || pos < end; }
    __device__ __forceinline__ PfSeg next(const PfPlan& plan) {
        PfSeg s;
        if (round < plan.rounds) {
            s.unit = round * gridDim.x + blockIdx.x;
            s.a = 0; s.e = PF_FRAC; s.tail = -1;
            ++round;
        } else {
            s.tail = pos / PF_FRAC;
            s.unit = plan.tail + s.tail;
            s.a = pos % PF_FRAC;
            pos = min(end, (s.tail + 1) * PF_FRAC);
            s.e = pos - s.tail * PF_FRAC;
        }
        return s;
    }
};

__device__ __forceinline__ int pf_rows_of(const SvlmAttendBatch& b, int ci, int n_q_arg) { return b.q_varlen ? b.q_cnt[ci] : n_q_arg; }

// Where a segment's rows lie, from the launch's arguments alone (warp-uniform).
struct PfRows {
    int ci, hk, n_q, m0, m_total;
    size_t q_row0, p_row0;   // first row in Q and out, in q_pos
    size_t head_row0;        // the head's first slot row in the K/V slabs
};
__device__ __forceinline__ PfRows pf_rows(const SvlmAttendBatch& b, const PfPlan& plan, int unit, int n_q_arg, int G, int layer0, int n_layers) {
    PfRows r;
    r.ci = 0;
    while (r.ci + 1 < b.n_caches && unit >= plan.off[r.ci + 1]) ++r.ci;
    r.n_q = pf_rows_of(b, r.ci, n_q_arg);
    r.m_total = r.n_q * G;
    const int R = (r.m_total + PF_ROWS - 1) / PF_ROWS, local = unit - plan.off[r.ci], t = pf_small_div(local, R);
    r.m0 = (local - t * R) * PF_ROWS;
    const int li = pf_small_div(t, b.kv_heads);
    r.hk = t - li * b.kv_heads;
    r.head_row0 = ((size_t)(layer0 + li) * b.kv_heads + r.hk) * b.n_slots;
    r.q_row0 = b.q_varlen ? (size_t)b.q_off[r.ci] : (size_t)(r.ci * n_layers + li) * n_q_arg;
    r.p_row0 = b.q_varlen ? (size_t)b.q_off[r.ci] : (size_t)r.ci * n_q_arg;
    return r;
}

// An entry of a cache's page list, ordinals relative to the first query token (those of long ago: some large negative number).
struct __align__(16) PfEntry {
    unsigned info;                 // page | lo << 14 | (hi - 1) << 21 | partly filled << 28 | ordinals one after another << 30
    int first, last, pad;
};
__device__ __forceinline__ PfEntry pf_entry(const int4& a, const longlong2& g, long long gid_q0) {
    PfEntry e;
    e.info = (unsigned)a.x | ((unsigned)a.y << 14) | ((unsigned)(a.z - 1) << 21) | ((unsigned)(a.y > 0 || a.z < SVLM_PAGE) << 28) |
             ((unsigned)(g.y - g.x == a.z - 1 - a.y) << 30);      // (ordinals grow with the offset)
    e.first = (int)max(g.x - gid_q0, -0x40000000ll);
    e.last = (int)max(g.y - gid_q0, -0x40000000ll);
    e.pad = 0;
    return e;
}
__device__ __forceinline__ PfEntry pf_load_entry(const SvlmAttendView& vw, int j, long long gid_q0) {
    const SvlmTile* tp = vw.tiles + j;
    const int4 a = ld_l2(reinterpret_cast<const int4*>(tp));
    return pf_entry(a, ld_l2(reinterpret_cast<const longlong2*>(&tp->min_gid)), gid_q0);
}

// What the cache's metadata says: fetched once per thread block, by warp 11, for the cache of the first segment.  All thread blocks
// begin at the same time, and with twelve warps of each reading the same few lines of L2 they waited for one another: 3900 cycles until
// the first page was known, 3300 now, and 11,700 until its S was there, 10,300 now (28/4 heads of 128, 524 tokens, many layers).
// Segments of other caches come at different times; there each warp looks by itself.
constexpr int PF_LIST = 96;
struct PfMeta {
    int ci, n_tiles;
    unsigned wait_limit;
    long long n_total, shift;
    PfEntry list[PF_LIST];         // the first entries of its page list
};

// What the metadata adds to a segment: its pages.
struct PfWork {
    const SvlmAttendView* vw;
    const PfEntry* list;           // the first PF_LIST entries, null: to be looked up
    int n_tiles, p0, n_proc;       // entries of the page list; of the pages that some row of the unit may see, [p0, p0 + n_proc)
    int rel_hi;                    // of the unit's last row's token
    long long gid_q0;              // ordinal of the first query token
    long long shift;
    unsigned wait_limit;
};
// What is known of a cache.
struct PfAsk {
    int first[PF_LIST / 32];       // of the first pages, relative to the first query token
    int n_tiles;
    long long n_total, shift;
    unsigned wait_limit;
};
// From its control block and its page list (the ordinals without waiting for their count, so that everything takes one round trip).
__device__ __forceinline__ PfAsk pf_ask(const SvlmAttendBatch& b, const PfRows& r) {
    PfAsk q;
    const SvlmAttendView& vw = b.view[r.ci];
    q.n_tiles = ld_l2(&vw.ctrl->n_tiles);
    q.n_total = ld_l2(&vw.ctrl->n_total);
    q.shift = ld_l2(&vw.ctrl->shift_total);
    q.wait_limit = ld_l2(&vw.ctrl->wait_limit);
    long long first[PF_LIST / 32];
#pragma unroll
    for (int k = 0; k < PF_LIST / 32; ++k) first[k] = ld_l2(&vw.tiles[min((int)(threadIdx.x & 31) + 32 * k, b.n_slots / SVLM_PAGE - 1)].min_gid);
#pragma unroll
    for (int k = 0; k < PF_LIST / 32; ++k) q.first[k] = (int)max(first[k] - (q.n_total - r.n_q), -0x40000000ll);
    return q;
}
__device__ __forceinline__ PfAsk pf_known(const PfMeta& meta) {
    PfAsk q;
    q.n_tiles = meta.n_tiles;
    q.n_total = meta.n_total;
    q.shift = meta.shift;
    q.wait_limit = meta.wait_limit;
#pragma unroll
    for (int k = 0; k < PF_LIST / 32; ++k) q.first[k] = meta.list[(threadIdx.x & 31) + 32 * k].first;
    return q;
}
__device__ __forceinline__ PfWork pf_work(const SvlmAttendBatch& b, const PfPlan& plan, const PfMeta& meta, const PfSeg& s, const PfRows& r, const PfAsk& q) {
    PfWork w;
    w.vw = &b.view[r.ci];
    w.list = r.ci == meta.ci ? meta.list : nullptr;
    w.n_tiles = q.n_tiles;
    w.gid_q0 = q.n_total - r.n_q;
    w.shift = q.shift;
    w.wait_limit = q.wait_limit;
    w.rel_hi = min(r.n_q - 1, pf_div(r.m0 + PF_ROWS - 1, plan));
    const int lane = threadIdx.x & 31;
    int n_act = 0;
#pragma unroll
    for (int k = 0; k < PF_LIST / 32; ++k) n_act += lane + 32 * k < w.n_tiles && q.first[k] <= w.rel_hi;
    for (int j = lane + PF_LIST; j < w.n_tiles; j += 32) n_act += ld_l2(&w.vw->tiles[j].min_gid) - w.gid_q0 <= w.rel_hi;
    n_act = __reduce_add_sync(0xffffffffu, n_act);
    w.p0 = s.a * n_act / PF_FRAC;
    w.n_proc = s.e * n_act / PF_FRAC - w.p0;
    return w;
}

// The softmax warpgroups keep what they know about their segment in shared memory: the page loop needs nearly all of
// their registers for the row of scores.
struct PfGroup {
    PfSeg seg;
    PfRows rows;
    PfWork w;
    PfWalk walk;
    int more;                // segments follow
    int known;               // the cache that the next five belong to (warp 11 sets the first one): a launch does not change its metadata
    int n_tiles;
    unsigned wait_limit;
    long long n_total, shift;
    int first[PF_LIST];      // smallest ordinals of the first pages of its list, relative to the first query token
    unsigned merge_later;    // blocks of columns of the first segment's unit that this CTA has to merge at the end
};

struct PfShared {            // control part of shared memory, behind the tiles
    unsigned long long full[PF_RING], empty[PF_RING];
    unsigned long long s_full[2], pv_done[2];
    unsigned tmem_base;
    int abort_flag;
    unsigned take[2];                      // per tile: blocks of columns of a cut unit that this CTA has to merge
    int leave[2];                          // its own ones are left to whoever comes last
    PfCut cut[2];                          // of the CTA's last segment, of its first one
    PfGroup group[2];
    int past[9][2];                        // per warp: PfPages
    PfMeta meta;
};
static_assert(sizeof(PfShared) <= 3072, "control block must fit behind the tiles");

// The columns of tensor memory (see the top).  Taking turns with one buffer of scores also keeps the two tiles half a page apart:
// with one each, which fit at head_dim 64, both do their exponentials at the same time, then neither (12/2 heads of 64, 4133
// tokens over 9200 keys 161 -> 177 us).
template <int D>
struct PfColumns {
    static constexpr unsigned S = 0;
    __device__ __forceinline__ static unsigned P(int g) { return 128 + g * 64; }
    __device__ __forceinline__ static unsigned O(int g) { return 256 + g * D; }
};
struct PfTmem { unsigned S, P, O; };      // of this thread's row

// One page of one row: S (128 fp32 columns, this thread's TMEM lane) -> P (64 columns of bf16 pairs), with a lazily
// moving reference maximum (O is rescaled only when the maximum grows by more than 2^8).  The whole row is loaded once
// and its columns given away (BAR_READ); the first half's maximum is taken while the second half is on its way.  Before
// P or O is touched, P V of the previous page has to be through (BAR_PV; it usually is, by then).  P goes out in chunks of 32 keys; once the exponentials of the third chunk are done, the first two chunks are
// certainly stored and are handed to the issuer (BAR_P1).  Of the blocks of 32 columns in mixed, the row sees those in
// [vlo, vlo + vlen): the blocks at the edge of what is visible, usually one or two (a second instance of this function for such
// pages, every column compared, had 28/4 heads, 2600 tokens over 2500 keys at 108 us a layer, this way it is 88; and it cost the
// other pages 2 %).
// All exponentials on the special-function unit, although it then has as many cycles of work as the tensor pipe: a polynomial
// on the FMA pipe for a quarter of them made a cold launch 5 % faster, but a chunk of many layers runs at the power limit,
// where its instructions cost clock (28 layers 2580 -> 2535 us, four layers of a long chunk 1740 -> 1718, one layer 105.0).
template <int D>
__device__ __forceinline__ void softmax_page(int g, const PfTmem& t, unsigned mixed, unsigned vlo, unsigned vlen, bool have_o, float& m_ref, float& l) {
    constexpr float c = D == 128 ? 0.12751743082459868f : 0.18033688011112042f;      // log2(e) / sqrt(D)
    auto visible = [&](int k) { return (unsigned)k - vlo < vlen; };
    float s[128];
    tmem_ld32(t.S, s);
    tmem_ld32(t.S + 32, s + 32);
    tmem_ld32(t.S + 64, s + 64);
    tmem_ld32(t.S + 96, s + 96);
    tmem_wait_ld<128>(s);
    tc_fence_before();
    bar_arrive(BAR_READ + g, 160);
    if (mixed) {
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
            if ((mixed >> ch) & 1) {
#pragma unroll
                for (int k = 32 * ch; k < 32 * ch + 32; ++k) s[k] = visible(k) ? s[k] : -INFINITY;
            }
    }
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int k = 0; k < 128; k += 2) mx[(k >> 1) & 3] = max3(mx[(k >> 1) & 3], s[k], s[k + 1]);
    const float mx_row = max3(fmaxf(mx[0], mx[1]), mx[2], mx[3]) * c;
    const bool grow = mx_row > m_ref + 8.f;
    const float m_new = grow ? mx_row : m_ref;
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    float corr = 1.f;
    bool wait_pv = have_o;
    if (__any_sync(0xffffffffu, grow)) {
        corr = grow ? exp2f(m_ref - m_use) : 1.f;   // m_ref = -inf gives 0
        if (have_o) {
            bar_sync(BAR_PV + g, 160);
            tc_fence_after();
            rescale_o(t.O, D, corr);
            wait_pv = false;
        }
    }
    const u64 c2 = pk64(c, c), nm2 = pk64(-m_use, -m_use);
    u64 sum[2] = {0ull, 0ull};
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
        unsigned pk[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k = ch * 32 + 2 * i;
            const u64 x = fma2(pk64(s[k], s[k + 1]), c2, nm2);
            float e0, e1;
            un64(x, e0, e1);
            e0 = ex2(e0);
            e1 = ex2(e1);
            sum[i & 1] = add2(sum[i & 1], pk64(e0, e1));
            pk[i] = pack2(e0, e1);
        }
        if (ch == 0 && wait_pv) {
            bar_sync(BAR_PV + g, 160);
            tc_fence_after();
        }
        if (ch == 2) {
            tmem_wait_st();
            tc_fence_before();
            bar_arrive(BAR_P1 + g, 160);
        }
        tmem_st16(t.P + ch * 16, pk);
    }
    float a0, a1, b0, b1;
    un64(sum[0], a0, a1);
    un64(sum[1], b0, b1);
    l = l * corr + ((a0 + a1) + (b0 + b1));
    m_ref = m_new;
    tmem_wait_st();
    tc_fence_before();
    bar_arrive(BAR_P2 + g, 160);
}


// A warp's walk over the pages of a segment, 32 entries of the cache's page list at a time, one per lane.
struct PfPages {
    int* past;               // in shared memory, since seldom wanted: entries looked at, pages seen among them
    unsigned left, info;     // pages of the window still to come; per lane: the entry's info, needs a mask << 28, causal << 29
    int first, at;           // per lane: ordinal of the page's first token, relative to the first query token; lane of the latest page
    __device__ __forceinline__ void begin(PfShared& sh) {
        past = sh.past[threadIdx.x >> 5];
        past[0] = 0;
        past[1] = 0;
        left = 0; info = 0; first = 0; at = 0;
    }
    // r_lo: rows from this token on are served; a page all of them see in full needs no mask
    __device__ __forceinline__ unsigned next(const PfWork& w, int r_lo) {
        while (left == 0) {
            const int base = past[0], seen = past[1];
            if (base >= w.n_tiles) break;
            const int lane = threadIdx.x & 31, j = min(base + lane, w.n_tiles - 1);
            const PfEntry e = w.list && base < PF_LIST ? w.list[j] : pf_load_entry(*w.vw, j, w.gid_q0);
            const bool vis = base + lane < w.n_tiles && e.first <= w.rel_hi;
            const unsigned causal = e.last > r_lo;
            info = e.info | (causal << 28) | (causal << 29);
            first = e.first;
            const unsigned all = __ballot_sync(0xffffffffu, vis);
            const int rank = seen + __popc(all & ((1u << lane) - 1));
            left = __ballot_sync(0xffffffffu, vis && rank >= w.p0 && rank < w.p0 + w.n_proc);
            __syncwarp();
            past[0] = base + 32;
            past[1] = seen + __popc(all);
            __syncwarp();
        }
        at = left ? __ffs(left) - 1 : 0;
        left &= left - 1;
        return __shfl_sync(0xffffffffu, info, at);
    }
    __device__ __forceinline__ int first_here() const { return __shfl_sync(0xffffffffu, first, at); }
};
// Rotates one 128-row tile of queries at q_pos - shift_total, rounds to bf16 and stores it K-major swizzled.  Called by
// the 128 threads of the tile's softmax warpgroup.  A work item is (row, 8 pairs): a 16-byte chunk of the row's low half
// with its partner of the high half; a thread keeps its chunk and takes every 128 / CH-th row.  The raw rows go to their
// places in shared memory asynchronously and are rotated there; meanwhile the factors of the tile's tokens (a token's G
// rows share them) are looked up, in batches without branches (look-ups that branched on the size of the position went
// out one by one).  This code runs once per unit, at the pace of the instruction fetch (4-8 cycles per instruction), so
// its loops are short: 15000 cycles when everything was unrolled.
template <int D>
struct PfTileRotation {
    static constexpr int HALF = D / 2, CH = D / 16, STEP = 128 / CH;      // chunks per half row; rows between a thread's items
    static constexpr int TPT = 128 / HALF;                                // tokens per pass of the 128 threads over the factors
    static constexpr int UN = 5;                                          // factors in flight per thread

    // element e of a row lives in block e/64, 16-byte chunk (e%64)/8, XOR-swizzled by row&7
    __device__ __forceinline__ static int at(int row, int e) { return (e / 64) * (128 * 128) + row * 128 + ((((e % 64) / 8) ^ (row & 7)) << 4); }

    __device__ __forceinline__ static void load(const PfPlan& plan, const PfRows& w, int g, int m, int G, int q_heads, const uint16_t* Q, unsigned char* sQ) {
        const int c8 = m % CH;
        const uint16_t* base = Q + (w.q_row0 * q_heads + w.hk * G) * D + c8 * 8;
        const unsigned lo = smem_u32(sQ) + at(m / CH, c8 * 8), hi = smem_u32(sQ) + at(m / CH, HALF + c8 * 8);      // (STEP is a multiple of 8: the swizzle stays)
#pragma unroll 2
        for (int u = 0; u < CH; ++u) {
            const int mg = w.m0 + g * 128 + m / CH + u * STEP;
            const bool live = mg < w.m_total;
            // row (token r, head h) lies at r * q_heads + h = r * (q_heads - G) + mg
            const uint16_t* src = live ? base + (size_t)(unsigned)(pf_div(mg, plan) * (q_heads - G) + mg) * D : base;
            const int n = live ? 16 : 0;                              // the rest is filled with zeros
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(lo + u * STEP * 128), "l"(src), "r"(n) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(hi + u * STEP * 128), "l"(src + HALF), "r"(n) : "memory");
        }
    }
    __device__ __forceinline__ static int axis_of(const SvlmAttendBatch& b, int pair) {
        return b.rope_mode == 0 ? 0 : (pair < b.sec_t ? 0 : (pair < b.sec_th ? 1 : 2));
    }
    // (cos, sin)(c * theta) for |c| < 2^16: two table entries, loaded without a branch (see svlm_rope.cuh)
    struct Near { float2 a, b; bool neg; };
    __device__ __forceinline__ static Near near_load(const float2* __restrict__ tab, int pair, int c) {
        const unsigned u = (unsigned)abs(c) & 0xffffu;
        return Near{__ldg(tab + (u & 255u) * HALF + pair), __ldg(tab + (256 + (u >> 8)) * HALF + pair), c < 0};
    }
    __device__ __forceinline__ static float2 near_value(const Near& n) {
        float2 r = svlm_cmul(n.a, n.b);
        if (n.neg) r.y = -r.y;
        return r;
    }
    __device__ __forceinline__ static bool is_near(long long c) { return c > -65536 && c < 65536; }

    // the tile's tokens and whether their factors fit the area
    __device__ __forceinline__ static bool staged(const PfPlan& plan, const PfRows& w, int g, int& t_lo, int& n_tok) {
        const int mt = w.m0 + g * 128;
        t_lo = min(w.n_q - 1, pf_div(mt, plan));
        n_tok = min(w.n_q - 1, pf_div(mt + 127, plan)) - t_lo + 1;
        return n_tok * (HALF * 8) <= PF_CS_BYTES;
    }
    // factors: per token HALF cosines, then HALF sines.  Eight consecutive lanes read eight values each at a time; the
    // 16-byte chunks are swizzled so that their halves fall into different banks
    __device__ __forceinline__ static int cs_at(int pair) { return (((pair >> 2) ^ ((pair >> 5) & 1)) << 2) | (pair & 3); }
    int c[UN];               // positions of the thread's first UN factors
    __device__ __forceinline__ void load_pos(const SvlmAttendBatch& b, const PfRows& w, const int* q_pos, int m, int t_lo, int n_tok, int tk0) {
        const int pw = b.rope_mode == 0 ? 1 : 3;
        const int* qp = q_pos + (w.p_row0 + t_lo) * pw + axis_of(b, m % HALF);
#pragma unroll
        for (int u = 0; u < UN; ++u) c[u] = ld_in(qp + (size_t)min(tk0 + u * TPT, n_tok - 1) * pw);
    }
    __device__ __forceinline__ void stage(const SvlmAttendBatch& b, const PfRows& w, long long shift, const int* q_pos, int m, int t_lo, int n_tok, float* s_cs) {
        const int pair = m % HALF;
        const float2* tab = reinterpret_cast<const float2*>(b.rope_tab);
        float* dst = s_cs + cs_at(pair);
        bool far = false;
#pragma unroll 1
        for (int tk0 = m / HALF; tk0 < n_tok; tk0 += TPT * UN) {
            Near v[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) {                                   // (the first batch of positions is here already)
                const long long cl = (long long)c[u] - shift;
                far |= !is_near(cl);
                v[u] = near_load(tab, pair, (int)cl);
            }
            load_pos(b, w, q_pos, m, t_lo, n_tok, tk0 + TPT * UN);           // beside the look-ups (of the last batch: its end once more)
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                const int tk = tk0 + u * TPT;
                const float2 f = near_value(v[u]);
                if (tk < n_tok) {
                    dst[(size_t)tk * 2 * HALF] = f.x;
                    dst[(size_t)tk * 2 * HALF + HALF] = f.y;
                }
            }
        }
        if (far) {                                     // native positions of a long stream
            const int pw = b.rope_mode == 0 ? 1 : 3;
            const int* qp = q_pos + (w.p_row0 + t_lo) * pw + axis_of(b, pair);
#pragma unroll 1
            for (int tk = m / HALF; tk < n_tok; tk += TPT) {
                const float2 f = svlm_rope_cs(tab, HALF, pair, (long long)ld_in(qp + (size_t)tk * pw) - shift, b.theta[pair]);
                dst[(size_t)tk * 2 * HALF] = f.x;
                dst[(size_t)tk * 2 * HALF + HALF] = f.y;
            }
        }
    }

    __device__ __forceinline__ static void rotate(const SvlmAttendBatch& b, const PfPlan& plan, const PfRows& w, long long shift, const int* q_pos, int g, int m,
                                                  int t_lo, bool from_stage, const float* s_cs, unsigned char* sQ) {
        const int c8 = m % CH;
#pragma unroll 1
        for (int u = 0; u < CH; ++u) {
            const int row = m / CH + u * STEP;
            const int tk = min(pf_div(w.m0 + g * 128 + row, plan), w.n_q - 1);
            uint4* plo = reinterpret_cast<uint4*>(sQ + at(row, c8 * 8));
            uint4* phi = reinterpret_cast<uint4*>(sQ + at(row, HALF + c8 * 8));
            const uint4 lo4 = *plo, hi4 = *phi;
            u64 cs[4], sn[4];                          // cosines and sines of the chunk's pairs, two and two
            if (from_stage) {
                const float* base = s_cs + (size_t)(tk - t_lo) * 2 * HALF;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(base + cs_at(c8 * 8 + 4 * j));
                    const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(base + HALF + cs_at(c8 * 8 + 4 * j));
                    cs[2 * j] = x.x; cs[2 * j + 1] = x.y;
                    sn[2 * j] = y.x; sn[2 * j + 1] = y.y;
                }
            } else {                                   // few heads per KV head: too many tokens for the area
                const float2* tab = reinterpret_cast<const float2*>(b.rope_tab);
                const int pw = b.rope_mode == 0 ? 1 : 3;
                const int* qp = q_pos + (w.p_row0 + tk) * pw;
                const long long p[3] = {ld_in(qp) - shift, ld_in(qp + pw / 2) - shift, ld_in(qp + pw - 1) - shift};
                Near v[8];
                bool far = false;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int a = axis_of(b, c8 * 8 + i);
                    const long long c = a == 0 ? p[0] : (a == 1 ? p[1] : p[2]);
                    far |= !is_near(c);
                    v[i] = near_load(tab, c8 * 8 + i, (int)c);
                }
                float2 f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] = near_value(v[i]);
                if (far) {
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const int a = axis_of(b, c8 * 8 + i);
                        const float2 x = svlm_rope_cs(tab, HALF, c8 * 8 + i, a == 0 ? p[0] : (a == 1 ? p[1] : p[2]), b.theta[c8 * 8 + i]);
#pragma unroll
                        for (int q = 0; q < 8; ++q) if (q == i) f[q] = x;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) { cs[j] = pk64(f[2 * j].x, f[2 * j + 1].x); sn[j] = pk64(f[2 * j].y, f[2 * j + 1].y); }
            }
            const unsigned* lw = reinterpret_cast<const unsigned*>(&lo4);
            const unsigned* hw = reinterpret_cast<const unsigned*>(&hi4);
            unsigned lo_o[4], hi_o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const u64 xl = pk64(__uint_as_float(lw[j] << 16), __uint_as_float(lw[j] & 0xffff0000u));
                const u64 xh = pk64(__uint_as_float(hw[j] << 16), __uint_as_float(hw[j] & 0xffff0000u));
                float a, c;
                un64(fma2(xl, cs[j], mul2(xh, sn[j] ^ 0x8000000080000000ull)), a, c);
                lo_o[j] = pack2(a, c);
                un64(fma2(xh, cs[j], mul2(xl, sn[j])), a, c);
                hi_o[j] = pack2(a, c);
            }
            *plo = make_uint4(lo_o[0], lo_o[1], lo_o[2], lo_o[3]);
            *phi = make_uint4(hi_o[0], hi_o[1], hi_o[2], hi_o[3]);
        }
    }
};

// End of the columns a row may see on a page with causal limits: stream ordinals grow with the offset, so it is the
// number of offsets whose ordinal (relative to the first query token) does not exceed the row's, found by bisection
// with shuffles over the page's 128 ordinals, four per lane (v; offsets below the valid range count as visible).
__device__ __forceinline__ int causal_end(const int (&v)[4], int r) {
    int L = 0;                                 // lanes all of whose four offsets are visible
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const int x = __shfl_sync(0xffffffffu, v[3], L + s - 1);
        if (x <= r) L += s;
    }
    {
        const int x = __shfl_sync(0xffffffffu, v[3], L);
        if (x <= r) L += 1;                    // (L was at most 31)
    }
    int n = 4 * L;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int x = __shfl_sync(0xffffffffu, v[k], L & 31);
        if (L < 32 && x <= r) ++n;
    }
    return n;
}

// 16 elements of an output row; wide: the launch's output begins at a multiple of 32 bytes.  A warp's store touches 32 rows, and
// what it costs is the rows, not the bytes: two 16-byte stores take twice as long as one of 32.
__device__ __forceinline__ void store_row16(uint16_t* dst, const float* o, bool wide) {
    unsigned v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = pack2(o[2 * k], o[2 * k + 1]);
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
    } else {
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

__device__ __forceinline__ uint16_t* out_row(uint16_t* out, const PfPlan& plan, const PfRows& w, int mg, int G, int q_heads, int D) {
    const int r = pf_div(mg, plan);      // row (token r, head h) lies at r * q_heads + h = r * (q_heads - G) + mg
    return out + (w.q_row0 * q_heads + w.hk * G + (size_t)(unsigned)(r * (q_heads - G) + mg)) * D;
}

// The scratch of a cut unit: CTA k's piece lies in k's first slot if it is k's first piece of the tail, else in the second.
template <int D>
struct PfSlot {
    unsigned char* base;
    __device__ __forceinline__ PfSlot(const PfPlan& plan, int tail, int k)
        : base(plan.slots + (size_t)(2 * k + (plan.x[k] >= tail * PF_FRAC ? 0 : 1)) * pf_slot_bytes<D>()) {}
    __device__ __forceinline__ float4* o(int g, int m) const { return reinterpret_cast<float4*>(base) + (size_t)g * 128 * (D / 4) + m; }   // + 128 per 4 columns
    __device__ __forceinline__ float2* ml(int g, int m) const { return reinterpret_cast<float2*>(base + (size_t)PF_ROWS * D * 4) + g * 128 + m; }
};

// Blocks of 16 columns of this CTA's piece of a cut unit into its slot (un-normalised, fp32).
template <int D>
__device__ __forceinline__ void publish_columns(const PfPlan& plan, int tail, int g, int m, unsigned tO, bool have_o, unsigned blocks) {
    if (!have_o) return;
    float4* po = PfSlot<D>(plan, tail, blockIdx.x).o(g, m);
#pragma unroll 1
    for (; blocks; blocks &= blocks - 1) {
        const int q = __ffs(blocks) - 1;
        float o[16];
        tmem_ld16(tO + q * 16, o);
        tmem_wait_ld<16>(o);
#pragma unroll
        for (int i = 0; i < 4; ++i) __stcg(po + (q * 4 + i) * 128, make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]));
    }
}

// The meeting of a unit's pieces, per tile.  One word counts arrivals (bits 0-7) and names the blocks of columns whose owners did
// not wait (16-23); a second one moves on when everybody is there.  A sharer has put down what the others need of its piece,
// counts itself in and waits for the rest, which the work split lets end at the same time: `polls` times at most.  If they
// are not there by then (their thread blocks may not even be running: another launch may hold the SMs) it puts down its own
// columns too, names them and leaves; whoever comes last merges them.  So nothing depends on a wait.  The last one clears the
// first word for the next launch.  Returns the blocks this CTA has to merge.
// Where nobody shares, the last one merges all, and keeps its piece in TMEM if the others are there already (last: the CTA's last
// segment, whose piece may stay there).
// Why wait, and how long: us per layer with its append, 28/4 heads of 128 over 9200 keys, 64 polls, 32, 16, 8 and (attention
// alone) none against 64: 69 tokens 48.6, 48.6, 53.9, 58.0 (46 and 38), 266 tokens 63.7, 63.9, 65.5, 67.1; over 43 shapes 1.059, 1.049,
// 1.015 and 1.001 times the speed of the last one merging by itself.  A block that waits keeps its SM from other streams: two
// equal streams' attention calls, nothing between them, run at 0.83-0.98 of that speed (0.91-0.96 with 8 polls), whole
// chunks of two streams at 0.93-1.03, unequal streams at 1.00-1.09, beside matrix products 0.97-1.00.  Waiting only for pieces
// that have been begun, or whose blocks started together, made no difference to any of these.
constexpr int PF_MEET_POLLS = 14;         // polls: the control block's limit >> this (64 by default, some 40 us)
template <int D>
__device__ __forceinline__ unsigned meet_pieces(PfShared& sh, const PfPlan& plan, int tail, const PfCut& cut, int g, int m, unsigned tO, float m_row, float l,
                                                bool have_o, bool last, unsigned polls) {
    constexpr unsigned ALL = (1u << (D / 16)) - 1;
    unsigned* word = plan.counters + (tail * 2 + g) * 2;
    if (last && cut.sharers == 0) {
        if (m == 0) {
            unsigned now;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(word) : "memory");
            sh.take[g] = (now & 255) == (unsigned)cut.pieces - 1 ? ALL : 0;
        }
        bar_sync(BAR_WG + g, 128);
        if (sh.take[g]) {
            if (m == 0) *word = 0;
            return ALL;
        }
    }
    unsigned turn = 0;                                       // of the second word: it cannot move before this CTA has arrived
    if (m == 0) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(turn) : "l"(word + 1) : "memory");
    __stcg(PfSlot<D>(plan, tail, blockIdx.x).ml(g, m), make_float2(have_o ? m_row : -INFINITY, l));
    publish_columns<D>(plan, tail, g, m, tO, have_o, ALL & ~cut.mine);
    bar_sync(BAR_WG + g, 128);
    if (m == 0) {
        __threadfence();
        unsigned before, take = 0;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(word) : "memory");
        bool all = (before & 255) == (unsigned)cut.pieces - 1;
        if (all) {
            take = cut.sharers ? cut.mine | before >> 16 : ALL;
            *word = 0;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(word + 1) : "memory");
        } else if (cut.mine) {
            for (unsigned p = 0; !all && p < polls; ++p) {
                unsigned now;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(word + 1) : "memory");
                all = now != turn;
            }
            take = all ? cut.mine : 0;
        }
        sh.take[g] = take;
        sh.leave[g] = cut.mine && !all;
    }
    bar_sync(BAR_WG + g, 128);
    if (sh.leave[g]) {
        publish_columns<D>(plan, tail, g, m, tO, have_o, cut.mine);
        bar_sync(BAR_WG + g, 128);
        if (m == 0) {
            __threadfence();
            unsigned before;
            asm volatile("atom.or.acq_rel.gpu.global.b32 %0, [%1], %2;" : "=r"(before) : "l"(word), "r"(cut.mine << 16) : "memory");
            const unsigned n = before & 255;
            const bool late = n == 0 || n == (unsigned)cut.pieces;      // the last one came in between: it has not seen the names, and clears or has cleared the word
            if (late) *word = 0;
            sh.take[g] = late ? cut.mine : 0;
        }
        bar_sync(BAR_WG + g, 128);
    }
    return sh.take[g];
}

// Some blocks of columns of a cut unit's output from its pieces, in the order of the pieces, whoever does it: the same bits
// every time.  This CTA's own piece may still be in TMEM (own: its last segment).  64 columns of the first two pieces are asked
// for at once, together with all pieces' (m, l), and the row's maximum and sum are taken once for all blocks.
template <int D>
__device__ __forceinline__ void merge_blocks(const PfPlan& plan, int tail, const PfCut& cut, unsigned take, const PfRows& w, int g, int m, int G, int q_heads,
                                             bool own, unsigned tO, float m_row, float l, bool have_o, uint16_t* __restrict__ out) {
    const int first = cut.first, last = cut.last, me = own ? (int)blockIdx.x : -1;
    const float m_own = have_o ? m_row : -INFINITY;
    auto after = [&](int k) {                                // the next piece, last + 1: none
        for (++k; k <= last && plan.x[k] >= plan.x[k + 1]; ++k) {}
        return k;
    };
    auto load = [&](int k, int q, int nb, float (&o)[64]) {  // nb blocks (of a piece without pages: left over from earlier, not used)
        if (k == me) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < nb && have_o) {
                    __syncwarp();
                    tmem_ld16(tO + (q + i) * 16, o + 16 * i);
                    tmem_wait_ld<16>(o + 16 * i);
                }
        } else {
            const float4* po = PfSlot<D>(plan, tail, k).o(g, m) + q * 4 * 128;
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (j < 4 * nb) {
                    const float4 v = ld_l2(po + j * 128);
                    o[4 * j] = v.x; o[4 * j + 1] = v.y; o[4 * j + 2] = v.z; o[4 * j + 3] = v.w;
                }
        }
    };
    auto ml_of = [&](int k) { return k == me ? make_float2(m_own, l) : ld_l2(PfSlot<D>(plan, tail, k).ml(g, m)); };
    const int mg = w.m0 + g * 128 + m;
    uint16_t* dst = out_row(out, plan, w, min(mg, w.m_total - 1), G, q_heads, D);
    const bool wide = !(reinterpret_cast<uintptr_t>(out) & 31);
    const int k2 = after(first);                             // (the first CTA's share is not empty, and a cut unit has two pieces at least)
    const float m1 = ml_of(first).x, m2 = ml_of(k2).x;
    float M = -INFINITY, inv = -1.f;
#pragma unroll 1
    while (take) {
        const int q = __ffs(take) - 1, nb = min(4, __ffs(~(take >> q)) - 1);
        take &= ~(((1u << nb) - 1) << q);
        float o1[64], o2[64];
        load(first, q, nb, o1);
        load(k2, q, nb, o2);
        if (inv < 0.f) {                                     // first time: the row's maximum and sum over all pieces, four in flight
            float L = 0.f;
#pragma unroll 1
            for (int k0 = first; k0 <= last; k0 += 4) {
                float2 ml[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = min(k0 + i, last);
                    ml[i] = ml_of(k);
                    if (k0 + i > last || plan.x[k] >= plan.x[k + 1]) ml[i].x = -INFINITY;
                }
                const float Mn = fmaxf(fmaxf(M, fmaxf(ml[0].x, ml[1].x)), fmaxf(ml[2].x, ml[3].x));
                if (Mn > -INFINITY) {
                    L *= exp2f(M - Mn);                      // M = -inf gives 0
#pragma unroll
                    for (int i = 0; i < 4; ++i) if (ml[i].x > -INFINITY) L += ml[i].y * exp2f(ml[i].x - Mn);
                    M = Mn;
                }
            }
            inv = L > 0.f ? 1.f / L : 0.f;
        }
        auto weight = [&](float mk) { return exp2f(mk - M) * inv; };
        const bool has1 = m1 > -INFINITY, has2 = m2 > -INFINITY;
        const float f1 = weight(m1), f2 = weight(m2);
#pragma unroll
        for (int c = 0; c < 64; ++c) {
            float x = has1 ? o1[c] * f1 : 0.f;
            if (has2) x += o2[c] * f2;
            o1[c] = x;
        }
#pragma unroll 1
        for (int k = after(k2); k <= last; k = after(k)) {
            const float mk = ml_of(k).x;
            load(k, q, nb, o2);
            if (mk > -INFINITY) {
                const float f = weight(mk);
#pragma unroll
                for (int c = 0; c < 64; ++c) o1[c] += o2[c] * f;
            }
        }
        if (mg < w.m_total) {
#pragma unroll
            for (int i = 0; i < 4; ++i) if (i < nb) store_row16(dst + (q + i) * 16, o1 + 16 * i, wide);
        }
    }
}

template <int D>
__global__ void __launch_bounds__(PF_THREADS, 1)
prefill_kernel(const __grid_constant__ SvlmAttendBatch b, const __grid_constant__ PfPlan plan, int layer0, int n_layers,
               const uint16_t* Q, const int* q_pos, int n_q_arg, int q_heads, uint16_t* __restrict__ out) {
    using Col = PfColumns<D>;
    constexpr int KB = D / 64;                 // 64-element (128-byte) blocks along d
    constexpr int TILE_BYTES = 128 * D * 2;    // one K or V page of one head, or one 128-row Q tile
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sQ = smem_raw;                             // [2 tiles][KB][128 rows][128 B]
    unsigned char* ring = sQ + 2 * TILE_BYTES;                // [stage][KB][128 keys][128 B]
    unsigned char* s_cs = ring + PF_RING * TILE_BYTES;        // [2 tiles] rotation factors
    PfShared& sh = *reinterpret_cast<PfShared*>(s_cs + 2 * PF_CS_BYTES);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = q_heads / b.kv_heads;
    volatile int* abort_flag = &sh.abort_flag;
    if (smem_u32(smem_raw) & 1023) {           // swizzled tiles need a 1024-byte aligned base; same in every CTA
        if (threadIdx.x == 0) atomicCAS(const_cast<int*>(&b.view[0].ctrl->status), 0, -4);   // SVLM_ERR_CUDA
        return;
    }

    // ---- set-up: barriers, TMEM ------------------------------------------------------
    if (threadIdx.x == 0) {
        for (int s = 0; s < PF_RING; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 2); }   // both issuers release a page
        for (int s = 0; s < 2; ++s) { mbar_init(&sh.s_full[s], 1); mbar_init(&sh.pv_done[s], 1); }
        sh.abort_flag = 0;
        mbar_init_fence();
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 32 || threadIdx.x == 64) {      // cut units: the last segment's, and the first one's where that is the end of one
        const int x0 = plan.x[blockIdx.x], x1 = plan.x[blockIdx.x + 1], which = threadIdx.x / 32 - 1;
        if (x0 < x1) sh.cut[which] = pf_cut(plan, (which ? x0 : x1 - 1) / PF_FRAC, blockIdx.x, D / 16);
    }
    // Set up while the predecessor ends (programmatic dependent launch): the roles also work out where their first segment lies,
    // which hangs on the launch's arguments only.  Everything read from here on may be the predecessor's work.
    // The wait comes before the trigger: a successor that starts early then finds all earlier work done.
    bool entered = false;
    auto enter = [&] {
        if (entered) return;
        entered = true;
        pdl_wait();
        pdl_launch_dependents();
        tc_fence_before();
        bar_sync(BAR_ALL, PF_THREADS);
        tc_fence_after();
    };

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        PfWalk walk;
        walk.begin(plan);
        bool ok = true;
        if (warp == 8) {
            // ================= TMA producer: K(0) K(1) V(0) K(2) V(1) ... V(n-1) through one ring, unit after unit =================
            unsigned item = 0;
            while (walk.more(plan)) {
                const PfSeg seg = walk.next(plan);
                const PfRows rows = pf_rows(b, plan, seg.unit, n_q_arg, G, layer0, n_layers);
                if (!entered) {
                    enter();
                    bar_sync(BAR_META, 128);
                }
                const PfWork w = pf_work(b, plan, sh.meta, seg, rows, rows.ci == sh.meta.ci ? pf_known(sh.meta) : pf_ask(b, rows));
                const void* tmK = w.vw->tmaps;
                const void* tmV = reinterpret_cast<const unsigned char*>(w.vw->tmaps) + 128;
                PfPages pages;
                pages.begin(sh);
                int y = 0, y_before = 0;
                for (int j = 0; j <= w.n_proc && ok; ++j) {
                    if (j < w.n_proc) y = (int)(rows.head_row0 + (size_t)(pages.next(w, 0) & 0x3FFF) * SVLM_PAGE);
                    if (lane == 0) {
#pragma unroll
                        for (int kv = 0; kv < 2; ++kv) {
                            if (kv ? j == 0 : j == w.n_proc) continue;
                            const unsigned st = item % PF_RING;
                            if (ok) ok = mbar_wait(&sh.empty[st], ((item / PF_RING) & 1) ^ 1, abort_flag, w.wait_limit);   // first pass: already free
                            if (!ok) break;
                            mbar_expect_tx(&sh.full[st], TILE_BYTES);
#pragma unroll
                            for (int kb = 0; kb < KB; ++kb)
                                tma_load_2d(ring + st * TILE_BYTES + kb * (128 * 128), kv ? tmV : tmK, kb * 64, kv ? y_before : y, &sh.full[st]);
                            ++item;
                        }
                    }
                    ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                    y_before = y;
                }
                if (!ok) break;
            }
        } else if (warp < 11) {
            // ================= MMA issuer of tile g =================
            // Per tile the order is S(0) | S(j+1) PV(j) | ...  The whole warp runs the loop (waits, descriptor arithmetic:
            // warp-uniform values the compiler can keep in uniform registers); one elected lane executes the tcgen05
            // instructions.  The number of named-barrier operations depends on the work list only, never on whether a wait
            // has run out, and so does their order: nobody arrives at a barrier again before the others have been there.
            //   BAR_READ of B's page j-1 -> S of A's page j -> BAR_S -> BAR_READ of A's page j -> S of B's page j -> ...
            //   BAR_P2 of a page -> its BAR_PV -> the next page's BAR_P1
            //   S of a page -> BAR_ASKED -> its BAR_S
            // Without a working wait everybody goes on along these lines, the issuers without issuing anything.  An issuer is past a product
            // only when the softmax has been at the earlier one's BAR_S, so BAR_ASKED keeps warp 11 from being there twice.
            const int g = warp - 9;
            const bool leader = elect_one();
            constexpr unsigned IDESC_S = make_idesc(128, 128, 0);
            constexpr unsigned IDESC_O = make_idesc(128, D, 1);
            // descriptors: the 14-bit start-address field counts 16-byte units, so moving inside a tile is an
            // addition to the low word (all tile addresses stay below the field's range: shared memory is 228 KB)
            unsigned tmem_s = 0, tmem_p = 0, tmem_o = 0;
            const unsigned long long dq = smem_desc(smem_u32(sQ + g * TILE_BYTES), 16, 1024);   // Q, K: K-major
            const unsigned long long dk = smem_desc(smem_u32(ring), 16, 1024);
            const unsigned long long dv = smem_desc(smem_u32(ring), 128 * 128, 1024);           // V: MN-major
            unsigned wait_limit = 0;
            auto wait_item = [&](int n) { if (ok) ok = __all_sync(0xffffffffu, mbar_wait_short(&sh.full[n % PF_RING], (n / PF_RING) & 1, abort_flag, wait_limit)); };
            auto issue_S = [&](unsigned n) {                        // S = Q K^T, K is ring item n
                const unsigned st = n % PF_RING;
                const unsigned long long b0 = dk + (unsigned)(st * TILE_BYTES >> 4);
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const unsigned off = ((ks / 4) * (128 * 128) + (ks % 4) * 32) >> 4;
                        tc_mma_ss(tmem_s, dq + off, b0 + off, IDESC_S, ks > 0);
                    }
                    tc_commit(&sh.s_full[g]);
                    tc_commit(&sh.empty[st]);
                }
                __syncwarp();
            };
            auto issue_PV = [&](unsigned n, int half, bool accumulate) {   // O += P V for 64 keys, V is ring item n
                const unsigned st = n % PF_RING;
                const unsigned long long b0 = dv + (unsigned)(st * TILE_BYTES >> 4);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {                   // 16 keys per MMA: A = 8 TMEM columns of bf16 pairs
                        const int ks = half * 4 + k;
                        tc_mma_ts(tmem_o, tmem_p + ks * 8, b0 + (unsigned)(ks * 2048 >> 4), IDESC_O, accumulate || k > 0);
                    }
                    if (half) { tc_commit(&sh.pv_done[g]); tc_commit(&sh.empty[st]); }
                }
                __syncwarp();
            };
            int item = 0;
            unsigned steps = 0, pvs = 0;
            auto step_S = [&](unsigned n) {
                // the order is A B A B ...: tile A's k-th S waits for B's k-1st to be read, tile B's for A's k-th
                if (g == 1 || steps > 0) bar_sync(BAR_READ + (g ^ 1), 160);
                if (ok) { tc_fence_after(); issue_S(n); }
                ++steps;
                bar_arrive(BAR_ASKED, 64);
            };
            while (walk.more(plan)) {
                const PfSeg seg = walk.next(plan);
                const PfRows rows = pf_rows(b, plan, seg.unit, n_q_arg, G, layer0, n_layers);
                if (!entered) {
                    enter();
                    bar_sync(BAR_META, 128);
                }
                const PfWork w = pf_work(b, plan, sh.meta, seg, rows, rows.ci == sh.meta.ci ? pf_known(sh.meta) : pf_ask(b, rows));
                const unsigned tmem = __shfl_sync(0xffffffffu, sh.tmem_base, 0);
                tmem_s = tmem + Col::S;
                tmem_p = tmem + Col::P(g);
                tmem_o = tmem + Col::O(g);
                wait_limit = w.wait_limit;
                const int n = w.n_proc;
                // ring items: K(0) K(1) V(0) K(2) V(1) ... K(n-1) V(n-2) V(n-1)
                auto k_of = [&](int j) { return j == 0 ? item : item + 2 * j - 1; };
                auto v_of = [&](int j) { return j + 1 < n ? item + 2 * j + 2 : item + 2 * j + 1; };
                if (n > 0) wait_item(item);
                bar_sync(BAR_Q + g, 160);
                if (n > 0) step_S(item);
                for (int j = 0; j < n; ++j) {
                    if (j + 1 < n) wait_item(k_of(j + 1));
                    wait_item(v_of(j));
                    if (j + 1 < n) step_S(k_of(j + 1));
                    bar_sync(BAR_P1 + g, 160);
                    if (ok) { tc_fence_after(); issue_PV(v_of(j), 0, j > 0); }
                    bar_sync(BAR_P2 + g, 160);
                    if (ok) {
                        tc_fence_after();
                        issue_PV(v_of(j), 1, true);
                        ok = __all_sync(0xffffffffu, mbar_wait_short(&sh.pv_done[g], pvs & 1, abort_flag, wait_limit));
                        tc_fence_after();
                        tc_fence_before();
                    }
                    bar_arrive(BAR_PV + g, 160);
                    ++pvs;
                }
                item += 2 * n;
            }
            if (g == 0 && steps > 0) bar_sync(BAR_READ + 1, 160);           // tile B's last one, behind which none comes
        } else {
            // ================= warp 11: says to the softmax that S is there =================
            // (A wait on an mbarrier costs a softmax warp ~300 cycles even when it is complete, a named barrier 40.)
            unsigned steps = 0;
            auto fetch_meta = [&](const PfRows& r) {
                const SvlmAttendView& vw = b.view[r.ci];
                int4 a[PF_LIST / 32];
                longlong2 g[PF_LIST / 32];
#pragma unroll
                for (int k = 0; k < PF_LIST / 32; ++k) {             // (pages that are not there: left over from earlier, not used)
                    const SvlmTile* tp = vw.tiles + min(lane + 32 * k, b.n_slots / SVLM_PAGE - 1);
                    a[k] = ld_l2(reinterpret_cast<const int4*>(tp));
                    g[k] = ld_l2(reinterpret_cast<const longlong2*>(&tp->min_gid));
                }
                const int n_tiles = ld_l2(&vw.ctrl->n_tiles);
                const long long n_total = ld_l2(&vw.ctrl->n_total), shift = ld_l2(&vw.ctrl->shift_total);
                const unsigned wait_limit = ld_l2(&vw.ctrl->wait_limit);
#pragma unroll
                for (int k = 0; k < PF_LIST / 32; ++k) {
                    const PfEntry e = pf_entry(a[k], g[k], n_total - r.n_q);
                    sh.meta.list[lane + 32 * k] = e;
                    sh.group[0].first[lane + 32 * k] = sh.group[1].first[lane + 32 * k] = e.first;
                }
                if (lane < 2) {
                    PfGroup& gr = sh.group[lane];
                    gr.known = r.ci; gr.n_tiles = n_tiles; gr.n_total = n_total; gr.shift = shift; gr.wait_limit = wait_limit;
                }
                if (lane == 0) { sh.meta.ci = r.ci; sh.meta.n_tiles = n_tiles; sh.meta.wait_limit = wait_limit; sh.meta.n_total = n_total; sh.meta.shift = shift; }
                __syncwarp();
            };
            while (walk.more(plan)) {
                const PfSeg seg = walk.next(plan);
                const PfRows rows = pf_rows(b, plan, seg.unit, n_q_arg, G, layer0, n_layers);
                if (!entered) {
                    enter();
                    fetch_meta(rows);
                    bar_sync(BAR_META, 128);
                    bar_arrive(BAR_S, 160);
                    bar_arrive(BAR_S + 1, 160);
                }
                const PfWork w = pf_work(b, plan, sh.meta, seg, rows, rows.ci == sh.meta.ci ? pf_known(sh.meta) : pf_ask(b, rows));
                for (int j = 0; j < w.n_proc; ++j, ++steps)
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        if (ok) ok = __all_sync(0xffffffffu, mbar_wait_short(&sh.s_full[g], steps & 1, abort_flag, w.wait_limit));
                        bar_sync(BAR_ASKED, 64);              // (nothing to wait for behind a wait that was met)
                        tc_fence_after();
                        tc_fence_before();
                        bar_arrive(BAR_S + g, 160);
                    }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // ================= softmax warpgroups: one thread per row of tile g =================
        const int g = warp >> 2, m = threadIdx.x & 127;
        PfTmem tm = {};
        bool ok = true;
        PfGroup& gr = sh.group[g];
        unsigned char* sQg = sQ + g * TILE_BYTES;
        float* cs_g = reinterpret_cast<float*>(s_cs + g * PF_CS_BYTES);
        float m_ref = -INFINITY, l = 0.f;
        if (m == 0) { gr.walk.begin(plan); gr.merge_later = 0; gr.more = gr.walk.more(plan); gr.seg.a = 0; gr.seg.e = PF_FRAC; }
        bar_sync(BAR_WG + g, 128);
        while (gr.more) {
            bar_sync(BAR_WG + g, 128);        // everybody is through with the previous segment's fields
            {
                PfWalk walk = gr.walk;
                const PfSeg seg = walk.next(plan);
                const PfRows rows = pf_rows(b, plan, seg.unit, n_q_arg, G, layer0, n_layers);
                // in the order in which the answers are needed: the memory system takes them one after another
                PfTileRotation<D> rot;
                int t_lo, n_tok;
                const bool staged = PfTileRotation<D>::staged(plan, rows, g, t_lo, n_tok);
                const bool start = !entered;
                enter();
                const unsigned lanes = sh.tmem_base + ((unsigned)((warp & 3) * 32) << 16);
                tm = {lanes + Col::S, lanes + Col::P(g), lanes + Col::O(g)};
                PfTileRotation<D>::load(plan, rows, g, m, G, q_heads, Q, sQg);
                if (start) {                  // warp 11 has put down what is known of the first segment's cache
                    if (staged) rot.load_pos(b, rows, q_pos, m, t_lo, n_tok, m / PfTileRotation<D>::HALF);
                    bar_sync(BAR_S + g, 160);
                }
                const bool fresh = rows.ci != gr.known;
                PfAsk ask;
                if (fresh) {
                    ask = pf_ask(b, rows);
                } else {
                    ask.n_tiles = gr.n_tiles; ask.n_total = gr.n_total; ask.shift = gr.shift; ask.wait_limit = gr.wait_limit;
#pragma unroll
                    for (int k = 0; k < PF_LIST / 32; ++k) ask.first[k] = gr.first[lane + 32 * k];
                }
                if (!start && staged) rot.load_pos(b, rows, q_pos, m, t_lo, n_tok, m / PfTileRotation<D>::HALF);
                const PfWork nw = pf_work(b, plan, sh.meta, seg, rows, ask);
                if (m == 0) { gr.seg = seg; gr.rows = rows; gr.w = nw; gr.more = walk.more(plan); }
                if (staged) rot.stage(b, rows, nw.shift, q_pos, m, t_lo, n_tok, cs_g);
                asm volatile("cp.async.wait_all;" ::: "memory");
                bar_sync(BAR_WG + g, 128);
                if (m == 0) gr.walk = walk;
                if (fresh && m < 32) {
                    if (m == 0) { gr.known = rows.ci; gr.n_tiles = ask.n_tiles; gr.n_total = ask.n_total; gr.shift = ask.shift; gr.wait_limit = ask.wait_limit; }
#pragma unroll
                    for (int k = 0; k < PF_LIST / 32; ++k) gr.first[m + 32 * k] = ask.first[k];
                }
                PfTileRotation<D>::rotate(b, plan, rows, nw.shift, q_pos, g, m, t_lo, staged, cs_g, sQg);
            }
            fence_proxy_async();              // the tile feeds the tensor core
            tc_fence_before();                // (the previous unit's accumulator has been read)
            const PfWork& w = gr.w;
            const int n_proc = w.n_proc;
            // (arrive: the issuer takes it from here.  A thread that would not be held up by the tensor pipe afterwards
            // has to sync instead, or it could arrive again before the issuer has seen the first time.)
            if (n_proc > 0) bar_arrive(BAR_Q + g, 160);
            else bar_sync(BAR_Q + g, 160);
            const int mt = gr.rows.m0 + g * 128;
            m_ref = -INFINITY;
            l = 0.f;
            const int r = min(pf_div(mt + m, plan), gr.rows.n_q - 1), r_lo = min(pf_div(mt, plan), gr.rows.n_q - 1);
            PfPages pages;
            pages.begin(sh);
            for (int j = 0; j < n_proc; ++j) {
                const unsigned pi = pages.next(w, r_lo);
                const bool masked = (pi >> 28) & 1;
                unsigned vlo = 0, vlen = SVLM_PAGE, mixed = 0;      // mixed: of which 32 columns some row of the warp does not see all
                if (masked) {
                    const int lo = (pi >> 14) & 127, hi = ((pi >> 21) & 127) + 1;
                    int end = hi;
                    if ((pi >> 30) & (pi >> 29) & 1) {     // the new chunk's tokens: causal.  One after another in the page: nothing to look up
                        end = min(hi, lo + max(0, r - pages.first_here() + 1));
                    } else if ((pi >> 29) & 1) {
                        const long long* gp = w.vw->slot_gid + (size_t)(pi & 0x3FFF) * SVLM_PAGE + 4 * lane;
                        const longlong2 ga = ld_in(reinterpret_cast<const longlong2*>(gp)), gb = ld_in(reinterpret_cast<const longlong2*>(gp) + 1);
                        const long long gv[4] = {ga.x, ga.y, gb.x, gb.y};
                        int v[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const long long rel = gv[k] - w.gid_q0;
                            const int o = 4 * lane + k;
                            v[k] = o < lo ? -1 : (o >= hi ? 0x7fffffff : (rel < 0 ? -1 : (int)min(rel, 0x7ffffffell)));
                        }
                        end = causal_end(v, r);
                    }
                    vlo = lo;
                    vlen = max(end, lo) - lo;
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) mixed |= (unsigned)!__all_sync(0xffffffffu, lo <= 32 * ch && end >= 32 * ch + 32) << ch;
                }
                bar_sync(BAR_S + g, 160);
                tc_fence_after();
                softmax_page<D>(g, tm, mixed, vlo, vlen, j > 0, m_ref, l);
            }
            if (n_proc > 0) bar_sync(BAR_PV + g, 160);
            tc_fence_after();
            ok = !*abort_flag;                // (of a wait that has run out nothing is known here: the barriers go on in their order)
            const bool have_o = ok && n_proc > 0;
            if (gr.seg.e - gr.seg.a == PF_FRAC) {                      // all of the unit's pages
                const float inv = l > 0.f ? 1.f / l : 0.f;
                const int mg = mt + m;
                uint16_t* dst = out_row(out, plan, gr.rows, min(mg, gr.rows.m_total - 1), G, q_heads, D);
                const bool wide = !(reinterpret_cast<uintptr_t>(out) & 31);
#pragma unroll 1
                for (int q4 = 0; q4 < D / 32; ++q4) {
                    float o[32];
                    if (have_o) {
                        tmem_ld32(tm.O + q4 * 32, o);
                        tmem_wait_ld<32>(o);
                    }
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = have_o ? o[i] * inv : 0.f;
                    if (mg < gr.rows.m_total) {
                        store_row16(dst + q4 * 32, o, wide);
                        store_row16(dst + q4 * 32 + 16, o + 16, wide);
                    }
                }
            } else if (gr.more) {                                      // the end of a unit that others have begun
                const unsigned take = meet_pieces<D>(sh, plan, gr.seg.tail, sh.cut[1], g, m, tm.O, m_ref, l, have_o, false, 0);
                if (m == 0) gr.merge_later = take;
            }
        }
        // What is left of cut units (outside the loop over segments: its code would cost the page loop registers).
        const bool have_o = ok && gr.w.n_proc > 0;
        unsigned take = 0;
        if (gr.seg.e - gr.seg.a < PF_FRAC)
            take = meet_pieces<D>(sh, plan, gr.seg.tail, sh.cut[0], g, m, tm.O, m_ref, l, have_o, true, gr.w.wait_limit >> PF_MEET_POLLS);
        bar_sync(BAR_WG + g, 128);
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const unsigned blocks = pass == 0 ? take : gr.merge_later;
            if (!blocks) continue;
            const int tail = (pass == 0 ? plan.x[blockIdx.x + 1] - 1 : (int)plan.x[blockIdx.x]) / PF_FRAC;
            const PfRows rows = pf_rows(b, plan, plan.tail + tail, n_q_arg, G, layer0, n_layers);
            merge_blocks<D>(plan, tail, sh.cut[pass], blocks, rows, g, m, G, q_heads, pass == 0, tm.O, m_ref, l, have_o, out);
        }
    }

    enter();                                   // (a thread block without work)

    // ---- teardown ------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (sh.abort_flag) {
        // Somebody gave up.  Copies already issued still land in this CTA's shared memory: give
        // every full-barrier a bounded chance to complete before the memory is released.
        if (threadIdx.x == 0) {
            for (int s = 0; s < PF_RING; ++s)
                for (unsigned p = 0; p < 2; ++p)
                    for (unsigned w = 0; w < (1u << 16) && !mbar_test(&sh.full[s], p); ++w) __nanosleep(32);
            for (int i = 0; i < b.n_caches; ++i) atomicCAS(const_cast<int*>(&b.view[i].ctrl->status), 0, -5);   // SVLM_ERR_TIMEOUT
        }
        __syncthreads();
    }
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem_base), "r"(512));
    }
}

template <int D>
constexpr size_t prefill_smem() { return (size_t)(2 + PF_RING) * 128 * D * 2 + 2 * PF_CS_BYTES + sizeof(PfShared); }

template <int D>
cudaError_t launch(const SvlmAttendBatch& b, int layer0, int n_layers, const uint16_t* Q, const int* q_pos, int n_q,
                   int q_heads, uint16_t* out, const SvlmPrefillLoad* held, void* counters, void* slots, cudaStream_t st) {
    cudaError_t e = svlm_allow_smem<prefill_kernel<D>>(prefill_smem<D>());
    if (e != cudaSuccess) return e;
    // the register split inside the kernel adds up only if the block is launched with exactly this many (the build sees to it)
    static const bool regs_ok = [] {
        cudaFuncAttributes a;
        return cudaFuncGetAttributes(&a, prefill_kernel<D>) == cudaSuccess && a.numRegs == PF_REGS_LAUNCH;
    }();
    if (!regs_ok) return cudaErrorLaunchOutOfResources;
    const int G = q_heads / b.kv_heads;
    const PfPlanned& planned = pf_plan(b, n_layers, n_q, G, held, std::min(svlm_sm_count(), PF_MAX_CTAS), slots != nullptr);
    const int grid = planned.grid;
    PfPlan plan = planned.plan;
    plan.counters = static_cast<unsigned*>(counters);
    plan.slots = static_cast<unsigned char*>(slots);
    return svlm_launch_chained(prefill_kernel<D>, dim3((unsigned)grid), dim3(PF_THREADS), prefill_smem<D>(), 1, st, b, plan, layer0, n_layers, Q, q_pos,
                               n_q, q_heads, out);
}

}  // namespace

bool svlm_prefill_supported(int n_pages, int group) { return n_pages <= PF_MAX_TILES && group >= 1; }

// The slots for pieces of units, where a cache is long enough for cutting to pay.
size_t svlm_prefill_slot_bytes(int n_pages, int head_dim) {
    if (n_pages < 3 * PF_MIN_PAGES) return 0;
    return (size_t)2 * std::min(svlm_sm_count(), PF_MAX_CTAS) * (head_dim == 128 ? pf_slot_bytes<128>() : pf_slot_bytes<64>());
}

cudaError_t svlm_launch_prefill(const SvlmAttendBatch& b, int layer0, int n_layers, int call_layers, const void* Q, const int* q_pos,
                                int n_q, int q_heads, void* out, const SvlmPrefillLoad* held, void* counters, void* slots, cudaStream_t st) {
    const SvlmPrefillSmall small = svlm_prefill_small_plan(b, call_layers, n_q, q_heads, held);
    if (small.tiles > 0) return svlm_launch_prefill_small(b, layer0, n_layers, Q, q_pos, n_q, q_heads, small, out, st);
    return b.head_dim == 128
        ? launch<128>(b, layer0, n_layers, (const uint16_t*)Q, q_pos, n_q, q_heads, (uint16_t*)out, held, counters, slots, st)
        : launch<64>(b, layer0, n_layers, (const uint16_t*)Q, q_pos, n_q, q_heads, (uint16_t*)out, held, counters, slots, st);
}
