// The chunk prefill's work split (svlm_prefill_sm100.cu): host code over plain numbers, no addresses.
#pragma once
#include <algorithm>
#include <cstring>

#include "svlm_dev.h"
#include "svlm_launch.h"

constexpr int PF_ROWS = 256;          // rows per unit
constexpr int PF_MAX_CTAS = 160;
// When units are cut: pages a CTA should have at least, and pieces per unit beyond which merging them costs what the shorter
// pieces save.  133 to 261 tokens over 1200 keys, 28/4 heads: 6 pages 31-33 us, 4 28.6-30; 69 tokens over 9200 keys: 18 pieces
// 56.6 us, 12 48.9, 8 44.8.
constexpr int PF_MIN_PAGES = 4;
constexpr int PF_MAX_PIECES = 9;
// What beginning a unit is reckoned as, in pages.  The cuts also decide against which reference maximum a row's weights are
// rounded to bf16 (a piece begins its own), so another number here changes outputs in their last places: it stays where it is
// unless that is worth it.  With 7, 270 chunk shapes (37 to 4133 tokens, 350 to 9200 keys, six head shapes, one to eight streams) take 0.3 % less on
// average, between 6 % less (16/2 heads, 133 tokens over 4800 keys 37.5 -> 35.3 us a layer) and 6 % more (199 tokens 34.4 -> 36.5); with 5 0.1 % less,
// between 5 % less and 10 % more.
constexpr int PF_PIECE = 10;
constexpr int PF_SNAP = 3;            // a cut closer than this many pages to a unit's end moves there: a piece costs ~3 pages of set-up

// The work split, made on the host: it needs the numbers of rows, and of the pages only an estimate (a unit's pages are
// cut at fractions), so the kernel starts on its first unit without waiting for anything on the device.
constexpr int PF_FRAC = 128;          // a unit's pages are cut at multiples of 1/128
struct PfPlan {
    int units;                        // all units of the launch
    int off[SVLM_MAX_BATCH + 1];      // first unit of every cache: (layer, KV head, row tile), row tile fastest
    int rounds;                       // whole units per CTA first: CTA i takes units i, grid + i, ...
    int tail;                         // the units from here on are dealt out by x
    unsigned short x[PF_MAX_CTAS + 1];// where each CTA's share of them begins, in 1/128 units
    unsigned g_magic, g_shift;        // n / G = n * g_magic >> g_shift for n < 2^31 (pf_div)
    unsigned* counters;               // filled in at the launch: [2 * PF_MAX_CTAS][2][2] per (tail unit, tile) arrivals, zero between launches, and a turn;
    unsigned char* slots;             //   [2 * grid] partial results
};
static_assert(2 * PF_MAX_CTAS * 2 * 2 * sizeof(unsigned) <= svlm_prefill_counter_bytes, "counters");

// How a cut unit of the tail is divided: its pieces lie with the thread blocks [first, last], those with an empty share left out;
// the ones that end in it (all of them but one that has other segments to come) share the merge, in blocks of 16 columns, the
// first `sharers` of them; 0: whoever comes last merges all.  Sharing pays from two that end together and eight blocks on: a
// thread block that shares puts its columns down before it knows whether it is the last, and the last one by itself has half
// as much to read at head_dim 64.  Us per layer with its append, shared and by the last one alone: head_dim 64, 12/2 heads, 524 tokens
// over 9200 keys 52.8, 50.5; 16/8 heads, 390 tokens over 1250 keys 35.8, 34.6; head_dim 128, 28/4 heads, 69 tokens over 9200 keys 47.0, 57 (the merge
// before there were shares), 524 tokens 85.7, 91; one that ends in the unit, 1500 tokens 177.9, 177.0.
struct PfCut {
    int first, last, pieces, sharers;
    unsigned mine;                    // blocks of columns that are thread block cta's, a bit each
};
__host__ __device__ inline PfCut pf_cut(const PfPlan& plan, int tail, int cta, int blocks) {
    const int u0 = tail * PF_FRAC, u1 = u0 + PF_FRAC;
    PfCut c;
    for (c.first = cta; plan.x[c.first] > u0; --c.first) {}
    for (c.last = cta; plan.x[c.last + 1] < u1; ++c.last) {}
    int ends = 0, me = blocks;
    c.pieces = 0;
    for (int k = c.first; k <= c.last; ++k) {
        if (plan.x[k] == plan.x[k + 1]) continue;
        ++c.pieces;
        if (plan.x[k + 1] > u1) continue;
        if (k == cta) me = ends;
        ++ends;
    }
    c.sharers = blocks < 8 || ends < 2 ? 0 : ends < blocks ? ends : blocks;
    c.mine = 0;
    for (int q = 0; q < blocks && me < c.sharers; ++q)
        if (q * c.sharers >= me * blocks && q * c.sharers < (me + 1) * blocks) c.mine |= 1u << q;
    return c;
}

// The work split of one launch (see the top of svlm_prefill_sm100.cu): whole units in rounds over the grid while at least two rounds
// are left, the rest cut so that every CTA ends at the same level.  Beginning a unit, or another piece of one, costs as
// much as PF_PIECE pages.  The numbers of pages are estimates; a wrong one costs balance only.  cut: there is
// scratch for the pieces of cut units.
inline void pf_make_plan(PfPlan& plan, const SvlmAttendBatch& b, int n_layers, int n_q, int G, const SvlmPrefillLoad* held, int max_ctas, bool cut, int& grid) {
    plan.g_shift = 31;                                     // 31 + ceil(log2 G): the reciprocal rounded up to 32 bits is off by less than 2^-31 of 1 / G
    while ((1ll << (plan.g_shift - 31)) < G) ++plan.g_shift;
    plan.g_magic = (unsigned)(((1ull << plan.g_shift) + G - 1) / G);
    plan.units = 0;
    long long all = 0;                                     // pages of the whole launch
    const int per_unit = n_layers * b.kv_heads;
    auto rows_of = [&](int i) { return b.q_varlen ? b.q_cnt[i] : n_q; };
    auto tiles_of = [&](int i) { return (rows_of(i) * G + PF_ROWS - 1) / PF_ROWS; };
    // expected pages of row tile rt of cache i: what is stored of the chunk behind its last row is invisible (of a chunk
    // longer than the windows little is stored)
    auto cost = [&](int i, int rt) {
        const int later = std::max(0, rows_of(i) - 1 - (rt * PF_ROWS + PF_ROWS - 1) / G);
        return std::max(1, held[i].pages - std::min(later, held[i].windows) / SVLM_PAGE);
    };
    for (int i = 0; i < b.n_caches; ++i) {
        plan.off[i] = plan.units;
        const int R = tiles_of(i);
        plan.units += per_unit * R;
        for (int rt = 0; rt < R; ++rt) all += (long long)per_unit * cost(i, rt);
    }
    plan.off[b.n_caches] = plan.units;
    const int U = plan.units;
    grid = (int)std::min<long long>(max_ctas, cut ? std::max<long long>(U, std::min<long long>(all / PF_MIN_PAGES, (long long)PF_MAX_PIECES * U)) : U);
    plan.rounds = std::max(0, U / grid - 1);
    plan.tail = plan.rounds * grid;
    const int nt = U - plan.tail;
    if (!cut || grid == U) {                               // whole units only
        for (int i = 0; i <= grid; ++i) plan.x[i] = (unsigned short)((long long)i * nt / grid * PF_FRAC);
        return;
    }
    // walk the units in order: what the whole rounds give each CTA, then the tail's costs
    int ci = 0, rt = 0, R = tiles_of(0), left = R * per_unit;    // position of unit u
    auto step = [&] {
        if (++rt == R) rt = 0;
        if (--left == 0 && ci + 1 < b.n_caches) { ++ci; R = tiles_of(ci); left = R * per_unit; rt = 0; }
    };
    int load[PF_MAX_CTAS] = {}, tail_cost[2 * PF_MAX_CTAS], most = 0, dearest = 1;
    for (int u = 0, at = 0; u < plan.tail; ++u) {
        load[at] += cost(ci, rt) + PF_PIECE;
        most = std::max(most, load[at]);
        if (++at == grid) at = 0;
        step();
    }
    for (int t = 0; t < nt; ++t) { tail_cost[t] = cost(ci, rt); dearest = std::max(dearest, tail_cost[t]); step(); }
    // deals the tail out at a level; true when everything has found its place
    auto deal = [&](double level) {
        int t = 0;
        double rem = tail_cost[0];
        for (int i = 0; i < grid; ++i) {
            plan.x[i] = (unsigned short)(t < nt ? t * PF_FRAC + (int)((tail_cost[t] - rem) / tail_cost[t] * PF_FRAC + 0.5) : nt * PF_FRAC);
            double room = level - load[i];
            while (t < nt && (room -= PF_PIECE) >= std::min((double)PF_SNAP, rem)) {
                double take = std::min(room, rem);
                if (rem - take < PF_SNAP) take = rem;                // no slivers
                room -= take;
                rem -= take;
                if (rem > 0) break;
                if (++t < nt) rem = tail_cost[t];
            }
        }
        return t >= nt;
    };
    // the lowest level that does, by bisection between the average and whole units for everybody
    double lo = ((double)all + (double)PF_PIECE * U) / grid, hi = most + (double)((nt + grid - 1) / grid) * (dearest + PF_PIECE) + PF_SNAP;
    for (int it = 0; it < 8 && hi - lo > 0.5; ++it) {
        const double mid = 0.5 * (lo + hi);
        (deal(mid) ? hi : lo) = mid;
    }
    deal(hi);
    plan.x[grid] = (unsigned short)(nt * PF_FRAC);
}

// What a plan is made from.  The layers of a chunk come one after another with the same numbers, and so do several streams
// that are served in turn, so a thread keeps its latest plans (making one takes microseconds).
struct PfPlanKey {
    int n_caches, kv_heads, n_layers, n_q, G, max_ctas, varlen, cut;
    int rows[SVLM_MAX_BATCH];
    SvlmPrefillLoad held[SVLM_MAX_BATCH];
};
struct PfPlanned {
    PfPlanKey key;
    PfPlan plan;
    int grid;                         // thread blocks; 0: empty entry
};
struct PfPlanMemo {
    static constexpr int N = 16;
    PfPlanned entry[N];
    int at, next;                     // the latest hit; the entry to replace
    long long made;
};
inline PfPlanMemo& pf_plan_memo() {
    thread_local PfPlanMemo memo = {};
    return memo;
}
// The reference is good until the thread's next call.
inline const PfPlanned& pf_plan(const SvlmAttendBatch& b, int n_layers, int n_q, int G, const SvlmPrefillLoad* held, int max_ctas, bool cut) {
    PfPlanKey key;
    std::memset(&key, 0, sizeof key);
    key.n_caches = b.n_caches; key.kv_heads = b.kv_heads; key.n_layers = n_layers; key.n_q = n_q; key.G = G;
    key.max_ctas = max_ctas; key.varlen = b.q_varlen; key.cut = cut;
    for (int i = 0; i < b.n_caches; ++i) { key.rows[i] = b.q_varlen ? b.q_cnt[i] : n_q; key.held[i] = held[i]; }
    PfPlanMemo& memo = pf_plan_memo();
    for (int k = 0; k < PfPlanMemo::N; ++k) {
        const int i = (memo.at + k) % PfPlanMemo::N;
        const PfPlanned& e = memo.entry[i];
        if (e.grid != 0 && std::memcmp(&e.key, &key, sizeof key) == 0) { memo.at = i; return e; }
    }
    PfPlanned& e = memo.entry[memo.next];
    memo.at = memo.next;
    memo.next = (memo.next + 1) % PfPlanMemo::N;
    ++memo.made;
    e.key = key;
    pf_make_plan(e.plan, b, n_layers, n_q, G, held, max_ctas, cut, e.grid);
    return e;
}
