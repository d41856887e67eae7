// Chunk-prefill attention for chunks of few rows (svlm_prefill_sm100.cu serves the rest): the smallest streams, and short
// chunks over short windows.  There the tensor-core kernel's time is not work but its fixed chain: tensor memory,
// register hand-over, 128-row prologue, one 128-key page after another through a single CTA, all of it code that runs once.
// Here a CTA takes 16 or 32 packed rows (row = (token, head in the GQA group)) of a KV head, its warps share the keys in
// sub-tiles of 32 (mma.sync, the rows being the M side), and meet once at the end; with long windows the keys are divided
// over a cluster of up to eight CTAs, which then merge through distributed shared memory.
// A warp fetches its own sub-tiles by TMA into two private stages; the first two are under way while the queries are
// rotated.  Every mbarrier wait is bounded; on expiry the CTA records SVLM_ERR_TIMEOUT, drains its copies and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_ptx.cuh"
#include "svlm_rope.cuh"
#include "svlm_tc.cuh"

namespace {

using namespace svlm_ptx;
using namespace svlm_tc;

constexpr int SM_TILE = 16;            // rows of an MMA
constexpr int SM_SUB = 32;            // keys per sub-tile: the box of the decode kernel's tensor maps
constexpr int SM_STAGES = 2;          // per warp
constexpr int SM_MAX_TILES = 512;
constexpr int SM_MAX_PARTS = 8;       // CTAs (a cluster) that divide the keys of the same rows
template <int D> constexpr int sm_warps = D == 128 ? 6 : 8;                     // (192 and 128 KB of stages)
template <int D> constexpr int sm_stage_bytes = 2 * SM_SUB * D * 2;             // K, then V
constexpr int SM_QPAD = 8;            // elements between the query rows: conflict-free ldmatrix
constexpr int SM_OPAD = 8;            // floats between the output rows of the merge

template <int MT> struct SmShared {
    unsigned long long full[8 * SM_STAGES];
    int abort_flag;
    int pad[3];
    float2 ml[8][SM_TILE * MT];       // per warp: each row's maximum and sum
    float2 cta_ml[SM_TILE * MT];      // the warps' together
    unsigned tile[SM_MAX_TILES];      // page | lo << 14 | (hi - 1) << 21 | causal << 28 | not visible to any row << 29
};
template <int D, int MT> constexpr size_t sm_smem =
    1024 + (size_t)sm_warps<D> * SM_STAGES * sm_stage_bytes<D> + (size_t)SM_TILE * MT * ((D + SM_OPAD) * 4 + (D + SM_QPAD) * 2) + sizeof(SmShared<MT>);
static_assert(sm_smem<128, 2> <= 227 * 1024 && SM_TILE * 2 * (128 + SM_OPAD) * 4 <= SM_STAGES * sm_stage_bytes<128> &&
              SM_TILE * 2 * (64 + SM_OPAD) * 4 <= SM_STAGES * sm_stage_bytes<64>, "stages, and the merge in them");

__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ unsigned pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned*>(&v);
}
// 16-byte chunk `chunk` of a key's row inside K or V of a stage (the layout of a 128-byte-swizzle box, 64 dims wide)
__device__ __forceinline__ int sm_off(int key, int chunk) { return (chunk >> 3) * (SM_SUB * 128) + key * 128 + (((chunk & 7) ^ (key & 7)) << 4); }

template <int D, int MT>
__global__ void __launch_bounds__(32 * sm_warps<D>, 1)
prefill_small_kernel(const __grid_constant__ SvlmAttendBatch b, int layer0, int n_layers, const uint16_t* Q,
                     const int* q_pos, int n_q_arg, int q_heads, int parts, uint16_t* __restrict__ out) {
    constexpr int ROWS = SM_TILE * MT;
    constexpr int W = sm_warps<D>, HALF = D / 2, KB = D / 64, STAGE = sm_stage_bytes<D>, V_AT = STAGE / 2;
    constexpr float c = D == 128 ? 0.12751743082459868f : 0.18033688011112042f;      // log2(e) / sqrt(D)
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float* cta_o = reinterpret_cast<float*>(ring + W * SM_STAGES * STAGE);           // [ROWS][D + pad]: this CTA's part of a cluster's output
    uint16_t* sQ = reinterpret_cast<uint16_t*>(cta_o + ROWS * (D + SM_OPAD));        // [ROWS][D + pad]
    SmShared<MT>& sh = *reinterpret_cast<SmShared<MT>*>(sQ + ROWS * (D + SM_QPAD));
    volatile int* abort_flag = &sh.abort_flag;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ci = blockIdx.z / n_layers, li = blockIdx.z % n_layers, hk = blockIdx.y;
    const int part = blockIdx.x % parts, m0 = blockIdx.x / parts * ROWS;              // (a cluster's CTAs share the rows and divide the keys)
    const SvlmAttendView& vw = b.view[ci];
    const int G = q_heads / b.kv_heads;
    const int n_q = b.q_varlen ? b.q_cnt[ci] : n_q_arg, m_total = n_q * G;
    if (tid == 0) {
        for (int s = 0; s < W * SM_STAGES; ++s) mbar_init(&sh.full[s], 1);
        sh.abort_flag = 0;
        mbar_init_fence();
    }
    pdl_wait();                       // the wait comes before the trigger: a successor that starts early finds all earlier work done
    pdl_launch_dependents();
    if (m0 >= m_total) return;        // (streams with chunks of different lengths)

    // ---- everything the prologue needs, in one round trip ----
    const int n_pages = b.n_slots / SVLM_PAGE;
    const int n_tiles = min(ld_l2(&vw.ctrl->n_tiles), SM_MAX_TILES);
    const long long gid_q0 = ld_l2(&vw.ctrl->n_total) - n_q, shift = ld_l2(&vw.ctrl->shift_total);
    const unsigned wait_limit = ld_l2(&vw.ctrl->wait_limit);
    const int r_lo = m0 / G, r_hi = min(n_q - 1, (m0 + ROWS - 1) / G);
    for (int i = tid; i < n_pages && (i < (int)blockDim.x || i < n_tiles); i += blockDim.x) {     // (the first ones without waiting for their count)
        const int4 a = ld_l2(reinterpret_cast<const int4*>(vw.tiles + i));
        const longlong2 g = ld_l2(reinterpret_cast<const longlong2*>(&vw.tiles[i].min_gid));
        const unsigned causal = g.y > gid_q0 + r_lo, unseen = g.x > gid_q0 + r_hi;
        sh.tile[i] = (unsigned)a.x | ((unsigned)a.y << 14) | ((unsigned)(a.z - 1) << 21) | (causal << 28) | (unseen << 29);
    }
    // a thread's query items: eight pairs of a row each
    constexpr int CH = D / 16, ITEMS = (ROWS * CH + 32 * W - 1) / (32 * W);
    uint4 lo4[ITEMS], hi4[ITEMS];
    int p[ITEMS][3];
    const size_t q_row0 = b.q_varlen ? (size_t)b.q_off[ci] : (size_t)(ci * n_layers + li) * n_q;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const int it = min(tid + u * 32 * W, ROWS * CH - 1), mg = min(m0 + it / CH, m_total - 1), r = mg / G;
        const uint16_t* src = Q + ((q_row0 + r) * q_heads + hk * G + (mg - r * G)) * D + (it % CH) * 8;
        lo4[u] = ld_in(reinterpret_cast<const uint4*>(src));
        hi4[u] = ld_in(reinterpret_cast<const uint4*>(src + HALF));
        const int pw = b.rope_mode == 0 ? 1 : 3;
        const int* qp = q_pos + ((b.q_varlen ? (size_t)b.q_off[ci] : (size_t)ci * n_q) + r) * pw;
        p[u][0] = ld_in(qp); p[u][1] = ld_in(qp + pw / 2); p[u][2] = ld_in(qp + pw - 1);
    }
    __syncthreads();

    // ---- this warp's sub-tiles: of all that hold visible keys, every (W * parts)-th ----
    const int mine = part * W + warp, of = W * parts;
    int base = 0, cur = 0, cnt = 0;
    unsigned own = 0;
    auto next = [&]() -> int {
        while (own == 0 && base < 4 * n_tiles) {
            const int q = base + lane;
            bool valid = false;
            if (q < 4 * n_tiles) {
                const unsigned t = sh.tile[q >> 2];
                const int k0 = (q & 3) * SM_SUB, lo = (t >> 14) & 127, hi = ((t >> 21) & 127) + 1;
                valid = !(t >> 29) && k0 < hi && k0 + SM_SUB > lo;
            }
            const unsigned all = __ballot_sync(0xffffffffu, valid);
            own = __ballot_sync(0xffffffffu, valid && (cnt + __popc(all & ((1u << lane) - 1))) % of == mine);
            cnt = (cnt + __popc(all)) % of;
            cur = base;
            base += 32;
        }
        if (own == 0) return -1;
        const int q = cur + __ffs(own) - 1;
        own &= own - 1;
        return q;
    };
    unsigned char* stages = ring + warp * SM_STAGES * STAGE;
    unsigned long long* full = sh.full + warp * SM_STAGES;
    const size_t head_row0 = ((size_t)(layer0 + li) * b.kv_heads + hk) * b.n_slots;
    const unsigned char* maps = reinterpret_cast<const unsigned char*>(vw.tmaps);
    int issued = 0, done = 0;
    auto fetch = [&](int q) {
        if (lane == 0) {
            unsigned char* dst = stages + (issued % SM_STAGES) * STAGE;
            unsigned long long* bar = full + issued % SM_STAGES;
            const int y = (int)(head_row0 + (size_t)(sh.tile[q >> 2] & 0x3FFF) * SVLM_PAGE + (q & 3) * SM_SUB);
            mbar_expect_tx(bar, STAGE);
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                tma_load_2d(dst + kb * (SM_SUB * 128), maps + 256, kb * 64, y, bar);
                tma_load_2d(dst + V_AT + kb * (SM_SUB * 128), maps + 384, kb * 64, y, bar);
            }
        }
        ++issued;
    };
    int qa = next(), qb = next();
    if (qa >= 0) fetch(qa);
    if (qb >= 0) fetch(qb);

    // ---- queries: rotated at q_pos - shift_total, rounded to bf16 ----
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const int it = tid + u * 32 * W, row = it / CH, c8 = it % CH;
        if (row >= ROWS) break;
        const float2* tab = reinterpret_cast<const float2*>(b.rope_tab);
        float2 f[8];
        bool far = false;
#pragma unroll
        for (int k = 0; k < 3; ++k) { const long long x = p[u][k] - shift; far |= x <= -65536 || x >= 65536; }
        auto pos_of = [&](int pair) {
            const int a = b.rope_mode == 0 ? 0 : (pair < b.sec_t ? 0 : (pair < b.sec_th ? 1 : 2));
            return (a == 0 ? p[u][0] : (a == 1 ? p[u][1] : p[u][2])) - shift;
        };
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = svlm_rope_cs_batched(tab, HALF, c8 * 8 + i, (int)pos_of(c8 * 8 + i));
        if (far) {                    // native positions of a long stream
#pragma unroll 1
            for (int i = 0; i < 8; ++i) {
                const float2 x = svlm_rope_cs(tab, HALF, c8 * 8 + i, pos_of(c8 * 8 + i), b.theta[c8 * 8 + i]);
#pragma unroll
                for (int q = 0; q < 8; ++q) if (q == i) f[q] = x;
            }
        }
        const unsigned lw[4] = {lo4[u].x, lo4[u].y, lo4[u].z, lo4[u].w}, hw[4] = {hi4[u].x, hi4[u].y, hi4[u].z, hi4[u].w};
        unsigned lo_o[4], hi_o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float x0 = __uint_as_float(lw[j] << 16), x1 = __uint_as_float(lw[j] & 0xffff0000u);
            const float y0 = __uint_as_float(hw[j] << 16), y1 = __uint_as_float(hw[j] & 0xffff0000u);
            const float2 f0 = f[2 * j], f1 = f[2 * j + 1];
            lo_o[j] = pack2(x0 * f0.x - y0 * f0.y, x1 * f1.x - y1 * f1.y);
            hi_o[j] = pack2(y0 * f0.x + x0 * f0.y, y1 * f1.x + x1 * f1.y);
        }
        uint16_t* dst = sQ + row * (D + SM_QPAD) + c8 * 8;
        *reinterpret_cast<uint4*>(dst) = make_uint4(lo_o[0], lo_o[1], lo_o[2], lo_o[3]);
        *reinterpret_cast<uint4*>(dst + HALF) = make_uint4(hi_o[0], hi_o[1], hi_o[2], hi_o[3]);
    }
    __syncthreads();

    const int g = lane >> 2, t = lane & 3, lm_i = lane >> 3, lm_r = lane & 7;
    auto q_fragment = [&](int mt, int ks, unsigned (&a)[4]) {
        ldmatrix_x4(a[0], a[1], a[2], a[3], sQ + (mt * SM_TILE + (lm_i & 1) * 8 + lm_r) * (D + SM_QPAD) + ks * 16 + (lm_i >> 1) * 8);
    };
    unsigned qf[MT == 1 ? D / 16 : 1][4];        // one tile's rows stay in registers, two tiles' are read as they are needed
    if constexpr (MT == 1) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) q_fragment(0, ks, qf[ks]);
    }
    int rel_q[MT][2];                             // tokens of the thread's rows, g and g + 8 of each tile
    float o[MT][D / 8][4], mx[MT][2], l[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            rel_q[mt][h] = min(n_q - 1, (m0 + mt * SM_TILE + g + 8 * h) / G);
            mx[mt][h] = -INFINITY;
            l[mt][h] = 0.f;
#pragma unroll
            for (int i = 0; i < D / 8; ++i) o[mt][i][2 * h] = o[mt][i][2 * h + 1] = 0.f;
        }
    bool ok = true;
    while (qa >= 0) {
        const unsigned ti = sh.tile[qa >> 2];
        const int k0 = (qa & 3) * SM_SUB, lo = (int)((ti >> 14) & 127) - k0, hi = (int)((ti >> 21) & 127) + 1 - k0;
        const bool causal = (ti >> 28) & 1;
        longlong2 gid[4];
        if (causal) {
            const long long* gp = vw.slot_gid + (size_t)(ti & 0x3FFF) * SVLM_PAGE + k0 + 2 * t;
#pragma unroll
            for (int nb = 0; nb < 4; ++nb) gid[nb] = ld_l2(reinterpret_cast<const longlong2*>(gp + nb * 8));
        }
        const int st = done % SM_STAGES;
        ok = mbar_wait(&full[st], (done / SM_STAGES) & 1, abort_flag, wait_limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const unsigned char* sk = stages + st * STAGE;
        const unsigned char* sv = sk + V_AT;
        float s[MT][4][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int nb = 0; nb < 4; ++nb)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[mt][nb][j] = 0.f;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            unsigned k4[2][4];
#pragma unroll
            for (int h = 0; h < 2; ++h)
                ldmatrix_x4(k4[h][0], k4[h][1], k4[h][2], k4[h][3], sk + sm_off(h * 16 + (lm_i >> 1) * 8 + lm_r, ks * 2 + (lm_i & 1)));
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                unsigned a4[4];
                if constexpr (MT == 1) { for (int i = 0; i < 4; ++i) a4[i] = qf[ks][i]; }
                else q_fragment(mt, ks, a4);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mma_bf16(s[mt][2 * h], a4[0], a4[1], a4[2], a4[3], k4[h][0], k4[h][1]);
                    mma_bf16(s[mt][2 * h + 1], a4[0], a4[1], a4[2], a4[3], k4[h][2], k4[h][3]);
                }
            }
        }
        if (causal || lo > 0 || hi < SM_SUB) {
#pragma unroll
            for (int nb = 0; nb < 4; ++nb)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int k = nb * 8 + 2 * t + j;
                    const bool in = k >= lo && k < hi;
                    const long long rel = causal ? (j ? gid[nb].y : gid[nb].x) - gid_q0 : -1;
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        if (!in || rel > rel_q[mt][0]) s[mt][nb][j] = -INFINITY;
                        if (!in || rel > rel_q[mt][1]) s[mt][nb][2 + j] = -INFINITY;
                    }
                }
        }
        unsigned pk[MT][4][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float corr[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v = -INFINITY;
#pragma unroll
                for (int nb = 0; nb < 4; ++nb) v = fmaxf(v, fmaxf(s[mt][nb][2 * h], s[mt][nb][2 * h + 1]));
                v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
                v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
                const float m_new = fmaxf(mx[mt][h], v * c), m_use = m_new == -INFINITY ? 0.f : m_new;
                corr[h] = ex2(mx[mt][h] - m_use);         // no key so far: 0
                mx[mt][h] = m_new;
                float sum = 0.f;
#pragma unroll
                for (int nb = 0; nb < 4; ++nb) {
                    const float e0 = ex2(fmaf(s[mt][nb][2 * h], c, -m_use)), e1 = ex2(fmaf(s[mt][nb][2 * h + 1], c, -m_use));
                    sum += e0 + e1;
                    pk[mt][nb][h] = pack2(e0, e1);
                }
                l[mt][h] = l[mt][h] * corr[h] + sum;      // (of the thread's columns: put together at the end)
            }
            if (done > 0 && __any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f)) {
#pragma unroll
                for (int i = 0; i < D / 8; ++i) { o[mt][i][0] *= corr[0]; o[mt][i][1] *= corr[0]; o[mt][i][2] *= corr[1]; o[mt][i][3] *= corr[1]; }
            }
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int db = 0; db < D / 16; ++db) {
                unsigned v4[4];
                ldmatrix_x4_trans(v4[0], v4[1], v4[2], v4[3], sv + sm_off(kk * 16 + (lm_i & 1) * 8 + lm_r, db * 2 + (lm_i >> 1)));
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_bf16(o[mt][2 * db], pk[mt][2 * kk][0], pk[mt][2 * kk][1], pk[mt][2 * kk + 1][0], pk[mt][2 * kk + 1][1], v4[0], v4[1]);
                    mma_bf16(o[mt][2 * db + 1], pk[mt][2 * kk][0], pk[mt][2 * kk][1], pk[mt][2 * kk + 1][0], pk[mt][2 * kk + 1][1], v4[2], v4[3]);
                }
            }
        __syncwarp();                             // the stage has been read
        ++done;
        qa = qb;
        qb = next();
        if (qb >= 0) fetch(qb);
    }

    // ---- the warps meet ----
    float* so = reinterpret_cast<float*>(stages);                                   // [ROWS][D + pad], in the warp's own stages
    if (ok) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = mt * SM_TILE + g + 8 * h;
                l[mt][h] += __shfl_xor_sync(0xffffffffu, l[mt][h], 1);
                l[mt][h] += __shfl_xor_sync(0xffffffffu, l[mt][h], 2);
                if (t == 0) sh.ml[warp][row] = make_float2(mx[mt][h], l[mt][h]);
#pragma unroll
                for (int i = 0; i < D / 8; ++i)
                    *reinterpret_cast<float2*>(so + row * (D + SM_OPAD) + i * 8 + 2 * t) = make_float2(o[mt][i][2 * h], o[mt][i][2 * h + 1]);
            }
    } else if (lane == 0) {
        // copies already issued still land in this CTA's shared memory: a bounded chance to complete before it is released
        for (int i = done; i < issued; ++i)
            for (unsigned w = 0; w < (1u << 16) && !mbar_test(&full[i % SM_STAGES], (i / SM_STAGES) & 1); ++w) __nanosleep(32);
    }
    __syncthreads();
    const bool gave_up = sh.abort_flag != 0;
    if (gave_up && tid == 0) atomicCAS(const_cast<int*>(&vw.ctrl->status), 0, -5);  // SVLM_ERR_TIMEOUT
    auto put = [&](int rw, int d8, const float (&acc)[8], float L) {
        const int r = (m0 + rw) / G;
        const float inv = L > 0.f ? 1.f / L : 0.f;
        uint16_t* dst = out + ((q_row0 + r) * q_heads + hk * G + (m0 + rw - r * G)) * D + d8 * 8;
        *reinterpret_cast<uint4*>(dst) = make_uint4(pack2(acc[0] * inv, acc[1] * inv), pack2(acc[2] * inv, acc[3] * inv),
                                                    pack2(acc[4] * inv, acc[5] * inv), pack2(acc[6] * inv, acc[7] * inv));
    };
    if (!gave_up)
        for (int it = tid; it < ROWS * (D / 8); it += 32 * W) {
            const int rw = it / (D / 8), d8 = it % (D / 8);
            if (m0 + rw >= m_total) break;
            float M = -INFINITY, L = 0.f, acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll
            for (int w = 0; w < W; ++w) M = fmaxf(M, sh.ml[w][rw].x);
            if (M > -INFINITY) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const float2 ml = sh.ml[w][rw];
                    const float f = ex2(ml.x - M);        // a warp without keys: 0
                    const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(ring + w * SM_STAGES * STAGE) + rw * (D + SM_OPAD) + d8 * 8);
                    const float4 a = src[0], e = src[1];
                    L += ml.y * f;
                    acc[0] += a.x * f; acc[1] += a.y * f; acc[2] += a.z * f; acc[3] += a.w * f;
                    acc[4] += e.x * f; acc[5] += e.y * f; acc[6] += e.z * f; acc[7] += e.w * f;
                }
            }
            if (parts == 1) put(rw, d8, acc, L);
            else {
                float4* dst = reinterpret_cast<float4*>(cta_o + rw * (D + SM_OPAD) + d8 * 8);
                dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
                dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
                if (d8 == 0) sh.cta_ml[rw] = make_float2(M, L);
            }
        }
    if (parts == 1) return;
    // ---- the cluster's CTAs meet: each puts its share of the outputs together from all of them (one that gave up too) ----
    __syncwarp();
    cluster_sync_all();
    for (int it = part * 32 * W + tid; it < ROWS * (D / 8); it += parts * 32 * W) {
        const int rw = it / (D / 8), d8 = it % (D / 8);
        if (m0 + rw >= m_total) break;
        float2 ml[SM_MAX_PARTS];
        float4 a[SM_MAX_PARTS], e[SM_MAX_PARTS];
        float M = -INFINITY, L = 0.f, acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll
        for (int k = 0; k < SM_MAX_PARTS; ++k) {
            ml[k] = make_float2(-INFINITY, 0.f);
            if (k >= parts) continue;
            const unsigned src = map_to_rank(cta_o + rw * (D + SM_OPAD) + d8 * 8, k);
            ml[k] = ld_cluster_v2(map_to_rank(&sh.cta_ml[rw], k));
            a[k] = ld_cluster_v4(src);
            e[k] = ld_cluster_v4(src + 16);
        }
#pragma unroll
        for (int k = 0; k < SM_MAX_PARTS; ++k) M = fmaxf(M, ml[k].x);
#pragma unroll
        for (int k = 0; k < SM_MAX_PARTS; ++k) {
            if (!(ml[k].x > -INFINITY)) continue;
            const float f = ex2(ml[k].x - M);
            L += ml[k].y * f;
            acc[0] += a[k].x * f; acc[1] += a[k].y * f; acc[2] += a[k].z * f; acc[3] += a[k].w * f;
            acc[4] += e[k].x * f; acc[5] += e[k].y * f; acc[6] += e[k].z * f; acc[7] += e[k].w * f;
        }
        put(rw, d8, acc, L);
    }
    __syncwarp();
    cluster_sync_all();               // nobody leaves while another still reads its shared memory
}

// most rows of q that a cache brings
int sm_rows(const SvlmAttendBatch& b, int n_q) {
    int rows = n_q;
    if (b.q_varlen) for (int i = 0; i < b.n_caches; ++i) rows = std::max(rows, b.q_cnt[i]);
    return rows;
}

template <int D, int MT>
cudaError_t launch(const SvlmAttendBatch& b, int layer0, int n_layers, const uint16_t* Q, const int* q_pos, int n_q, int q_heads, int parts,
                   uint16_t* out, cudaStream_t st) {
    cudaError_t e = svlm_allow_smem<prefill_small_kernel<D, MT>>(sm_smem<D, MT>);
    if (e != cudaSuccess) return e;
    const int tiles = (sm_rows(b, n_q) * (q_heads / b.kv_heads) + SM_TILE * MT - 1) / (SM_TILE * MT);
    return svlm_launch_chained(prefill_small_kernel<D, MT>, dim3(tiles * parts, b.kv_heads, b.n_caches * n_layers), dim3(32 * sm_warps<D>), sm_smem<D, MT>,
                               parts, st, b, layer0, n_layers, Q, q_pos, n_q, q_heads, parts, out);
}

}  // namespace

// Whether a launch is this kernel's business, and in which shape.  Measured (us per launch, head size 128 and 64): a CTA
// takes a fixed part and a part per 1000 keys, both listed below; a launch takes that for every round of CTAs, and there
// are as many at once as clusters of that size find room for (4: 112 fit, 136 do not; 8: 80 fit, 128 do not).  Two tiles
// per CTA cost more than one, but less than a second round.  The tensor-core kernel takes what is estimated at the end,
// more with many rows, and that again for every 148 units of 256 rows; so the few rows are here, up to long windows, and more rows with short ones.  The
// tensor-core kernel -> this one: 4 heads of 64, 37 tokens, 240 keys: 17.3 -> 4.8; 28/4 heads of 128: 37 tokens, 180 keys
// 20 -> 7; 133 tokens, 700 keys 25 -> 16; 37 tokens, 9100 keys 48 -> 37.  133 tokens over 9100 keys stay with the
// tensor-core kernel (48 against 97 here).
SvlmPrefillSmall svlm_prefill_small_plan(const SvlmAttendBatch& b, int call_layers, int n_q, int q_heads, const SvlmPrefillLoad* held) {
    struct Shape { int tiles, parts, at_once; float fixed[2], per_key[2]; };       // [head size 128, 64]
    static constexpr Shape shapes[] = {{1, 1, 148, {6.0f, 4.4f}, {6.1f, 3.6f}}, {1, 2, 144, {7.0f, 5.8f}, {3.3f, 1.95f}},
                                       {1, 4, 112, {7.4f, 6.3f}, {1.75f, 1.05f}}, {1, 8, 80, {7.5f, 6.4f}, {1.1f, 0.7f}},
                                       {2, 1, 148, {9.5f, 5.8f}, {10.1f, 5.0f}}};
    int pages = 1;
    for (int i = 0; i < b.n_caches; ++i) pages = std::max(pages, held[i].pages);
    const int at = b.head_dim == 128 ? 0 : 1;
    const long long rows = (long long)sm_rows(b, n_q) * (q_heads / b.kv_heads);
    const float keys = pages * (SVLM_PAGE / 1000.f);
    float best = at == 0 ? std::min(14.f + 1.4f * pages, 21.f + 0.35f * pages) : std::min(12.5f + 1.2f * pages, 22.f + 0.12f * pages);
    const long long units = (rows + 255) / 256 * b.kv_heads * b.n_caches * call_layers;
    best *= std::max(1.f, units / 148.f);
    SvlmPrefillSmall how = {0, 1};
    for (const Shape& s : shapes) {
        const long long ctas = (rows + SM_TILE * s.tiles - 1) / (SM_TILE * s.tiles) * s.parts * b.kv_heads * b.n_caches * call_layers;
        const float t = (float)((ctas + s.at_once - 1) / s.at_once) * (s.fixed[at] + s.per_key[at] * keys);
        if (t < best) { best = t; how = {s.tiles, s.parts}; }
    }
    return how;
}

cudaError_t svlm_launch_prefill_small(const SvlmAttendBatch& b, int layer0, int n_layers, const void* Q, const int* q_pos, int n_q,
                                      int q_heads, SvlmPrefillSmall how, void* out, cudaStream_t st) {
    auto* go = b.head_dim == 128 ? (how.tiles == 2 ? launch<128, 2> : launch<128, 1>) : (how.tiles == 2 ? launch<64, 2> : launch<64, 1>);
    return go(b, layer0, n_layers, (const uint16_t*)Q, q_pos, n_q, q_heads, how.parts, (uint16_t*)out, st);
}
