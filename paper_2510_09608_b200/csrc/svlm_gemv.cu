// Projections of a few tokens at a time (decode): Y = X W^T for n <= 16 rows of X.  With so few rows the
// work is reading W once, so these are bandwidth kernels; the arithmetic rides on mma.sync, with the tokens as (mostly
// empty) M rows, because it takes a fifth of the instructions of unpacking and multiplying on the FMA pipe.  They serve
// svlm_out_proj for small n, on both sides of the decode step: [q | k | v] = W_qkv x before svlm_decode_step, W_o a after it.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_ptx.cuh"

namespace {

__device__ __forceinline__ void mma_bf16_16816(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Up to 4 tokens.  Block i owns a run of output rows and walks it in stages of eight rows x KS elements of K; a stage
// belongs to one warp, which computes the eight rows' partial dot products with mma.sync (a lane's 16 bytes of a W row are
// the B fragments of two MMAs: a dot product does not care in which order k is summed).  A warp's stages come in turn
// through a shared-memory slot (cp.async.bulk) and through registers, so there are no hand-offs between warps.  Partial
// sums wait in shared memory and are added in the order of K at the end: the same bits every time.
// The weights depend on nothing earlier in the stream: while the predecessor still runs (programmatic dependent launch)
// the block fills slots and registers (135 KB) and asks for the rest of its rows into L2; behind the wait only the token
// vectors come from the predecessor.  Sized to fit beside a decode step's CTA: a decoder's chain of projections and decode
// steps otherwise leaves HBM idle while a decode step combines its partial results.  Chain of 3584 -> 4608, decode step,
// 3584 -> 3584 (77.6 MB): 28.9 us per layer with two blocks per SM that fetched one row per warp ahead, 24.5 with slots
// only (each refill is a round trip to L2 of over 1 us), 23.3 with both, 22.7 without selects where stages are whole (FORM below) and with
// the weights marked as read once (l2_read_once): two tokens of that chain through 28 layers, both policies on the present code, 1297 -> 1274 us;
// one layer's weights, which stay in L2, take the same time with either (2048 x 6144 4.77 us, 4096 x 4096 6.36).
constexpr int GV_THREADS = 256;
constexpr int GT_WARPS = 8;
constexpr int GT_SLOTS = GT_WARPS;      // one per warp
constexpr int GT_KS = 512;              // most elements of K in a stage
constexpr int GT_KB = GT_KS / 32;       // k-blocks of 32
constexpr int GT_ROW = GT_KS * 2 + 64;  // bytes between a stage's rows: two rows' 64-byte pieces fill the 32 banks
constexpr int GT_MAX_STAGES = 64;       // stages of one block (partial sums in shared memory); more rows take more blocks
constexpr int GT_PAD = 32;              // elements between the token rows, for the same reason
constexpr int GT_MAX_X = 100 * 1024;    // bytes of the token rows

struct __align__(16) GtShared {
    float part[GT_MAX_STAGES][4][8];    // [stage][token][row]
    unsigned long long full[GT_SLOTS];
    int abort_flag;
};
static_assert(sizeof(GtShared) % 16 == 0 && (GT_SLOTS * 8 * GT_ROW) % 128 == 0 && GT_ROW % 16 == 0 && GT_PAD % 8 == 0, "16-byte accesses");

__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, void* bar, unsigned long long policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(svlm_ptx::smem_u32(dst)), "l"(src), "r"(bytes), "r"(svlm_ptx::smem_u32(bar)), "l"(policy) : "memory");
}
// (the read-only path: weights are written by no kernel)
__device__ __forceinline__ uint4 ld_weights(const uint4* p, unsigned long long policy) {
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
    return v;
}

// parts: stages per group of eight rows; ks: elements of K per stage (a multiple of 64; the last part may be shorter)
// FORM: which of the stages are GT_KS long.  Each has its own kernel, since a launch of 2 to 8 us notices the fetching of code that it does
// not run (one token, weights from HBM, us, one kernel for all: 3584 x 512 2.87, this way 2.49; 2048 x 6144 5.98, 5.33):
//   GT_WHOLE  all (in_dim a multiple of GT_KS): nothing to choose or to look at
//   GT_MIXED  all but the last: a uniform branch.  4544 x 4096 10.5 with selects, 9.8 this way
//   GT_SHORT  none: selects.  1344 x 4096 3.63 with branches, 3.1 this way; 3136 x 4096 7.9, 7.3
enum GtForm { GT_WHOLE, GT_MIXED, GT_SHORT };
template <int FORM>
__global__ void __launch_bounds__(GT_WARPS * 32, 2) gemv_few_kernel(const uint16_t* X, const uint16_t* __restrict__ W,
                                                                 uint16_t* __restrict__ Y, int n, int in_dim, int out_dim, int parts,
                                                                 int ks, SvlmCtrl* ctrl) {
    using namespace svlm_ptx;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* ring = smem_raw;                                         // [slot][8 rows][GT_ROW]
    GtShared& sh = *reinterpret_cast<GtShared*>(ring + GT_SLOTS * 8 * GT_ROW);
    uint16_t* sx = reinterpret_cast<uint16_t*>(&sh + 1);                    // [n][in_dim + GT_PAD]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, kq = lane & 3;
    const int r0 = (int)((long long)out_dim * blockIdx.x / gridDim.x), r1 = (int)((long long)out_dim * (blockIdx.x + 1) / gridDim.x);
    const int n_stages = (r1 - r0 + 7) / 8 * parts;
    volatile int* abort_flag = &sh.abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < GT_SLOTS; ++i) mbar_init(&sh.full[i], 1);
        sh.abort_flag = 0;
        mbar_init_fence();
    }
    __syncthreads();
    pdl_launch_dependents();
    const unsigned long long once = l2_read_once();
    // stage s: rows from r0 + (s / parts) * 8, elements from (s % parts) * ks.  A warp's stages are warp, warp + GT_WARPS, ...:
    // those at even places come through its slot, those at odd places through registers.
    auto fetch = [&](int s) {
        if (s >= n_stages) return;
        const int row = r0 + s / parts * 8, k0 = s % parts * ks, rows = min(8, r1 - row), len = min(ks, in_dim - k0) * 2;
        void* bar = &sh.full[warp];
        if (lane == 0) mbar_expect_tx(bar, rows * len);
        __syncwarp();
        if (lane < rows) bulk_load(ring + (warp * 8 + lane) * GT_ROW, W + (size_t)(row + lane) * in_dim + k0, len, bar, once);
    };
    uint4 wr[GT_KB];
    auto load_regs = [&](int s) {
        if (s >= n_stages) return;
        const int row = min(r0 + s / parts * 8 + g, r1 - 1), k0 = s % parts * ks, kbs = min(ks, in_dim - k0) / 32;
        const uint4* p = reinterpret_cast<const uint4*>(W + (size_t)row * in_dim + k0) + kq;
        if (FORM == GT_SHORT) {
#pragma unroll
            for (int kb = 0; kb < GT_KB; ++kb) wr[kb] = kb < kbs ? __ldg(p + 4 * kb) : make_uint4(0, 0, 0, 0);
        } else if (FORM == GT_WHOLE || kbs == GT_KB) {
#pragma unroll
            for (int kb = 0; kb < GT_KB; ++kb) wr[kb] = ld_weights(p + 4 * kb, once);
        } else {
#pragma unroll
            for (int kb = 0; kb < GT_KB; ++kb)
                if (kb < kbs) wr[kb] = ld_weights(p + 4 * kb, once);
        }
    };
    fetch(warp);
    load_regs(warp + GT_WARPS);
    {   // whole groups behind those: rows lie one after another
        const int row = min(r0 + 2 * GT_WARPS / parts * 8, r1);
        const char* p = reinterpret_cast<const char*>(W + (size_t)row * in_dim);
        const size_t bytes = (size_t)(r1 - row) * in_dim * 2;               // a multiple of 128
        for (size_t o = (size_t)threadIdx.x * 2048; o < bytes; o += GT_WARPS * 32 * 2048)
            asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(p + o), "r"((unsigned)min((size_t)2048, bytes - o)), "l"(once) : "memory");
    }
    const unsigned wait_limit = ld_l2(&ctrl->wait_limit);                  // written at creation only, never by a kernel
    pdl_wait();
    const int row16 = in_dim / 8;                                           // 16-byte chunks of a token row
    for (int i = threadIdx.x; i < n * row16; i += GT_WARPS * 32)
        *reinterpret_cast<uint4*>(sx + (size_t)(i / row16) * GT_PAD + (size_t)i * 8) = ld_l2(reinterpret_cast<const uint4*>(X) + i);
    __syncthreads();
    const bool live = g < n;                                                // (the other rows of the MMA hold the last token once more: nobody reads their sums)
    const uint16_t* xrow = sx + (size_t)min(g, n - 1) * (in_dim + GT_PAD) + kq * 8;
    auto put = [&](int s, const float (&c)[4][4]) {
        if (live)
            *reinterpret_cast<float2*>(&sh.part[s][g][2 * kq]) = make_float2((c[0][0] + c[1][0]) + (c[2][0] + c[3][0]), (c[0][1] + c[1][1]) + (c[2][1] + c[3][1]));
    };
    unsigned phase = 0;
    for (int s = warp; s < n_stages; s += 2 * GT_WARPS) {
        const int s1 = s + GT_WARPS;
        if (s1 < n_stages) {
            const int k0 = s1 % parts * ks, kbs = min(ks, in_dim - k0) / 32;
            const uint16_t* xs = xrow + k0;
            float c[4][4] = {};                                             // four independent chains
            auto block = [&](int kb) {
                const uint4 a = *reinterpret_cast<const uint4*>(xs + kb * 32);
                mma_bf16_16816(c[2 * (kb & 1)], a.x, 0u, a.y, 0u, wr[kb].x, wr[kb].y);
                mma_bf16_16816(c[2 * (kb & 1) + 1], a.z, 0u, a.w, 0u, wr[kb].z, wr[kb].w);
            };
            if (FORM == GT_SHORT) {                                         // (written out: with the selects in `block` 1344 x 4096 takes 3.7 us)
                const int last = kbs - 1;
#pragma unroll
                for (int kb = 0; kb < GT_KB; ++kb) {
                    uint4 a = *reinterpret_cast<const uint4*>(xs + min(kb, last) * 32);
                    if (!live || kb > last) a = make_uint4(0, 0, 0, 0);
                    mma_bf16_16816(c[2 * (kb & 1)], a.x, 0u, a.y, 0u, wr[kb].x, wr[kb].y);
                    mma_bf16_16816(c[2 * (kb & 1) + 1], a.z, 0u, a.w, 0u, wr[kb].z, wr[kb].w);
                }
            } else if (FORM == GT_WHOLE || kbs == GT_KB) {
#pragma unroll
                for (int kb = 0; kb < GT_KB; ++kb) block(kb);
            } else {
#pragma unroll
                for (int kb = 0; kb < GT_KB; ++kb)
                    if (kb < kbs) block(kb);
            }
            load_regs(s1 + 2 * GT_WARPS);
            put(s1, c);
        }
        const bool ok = mbar_wait(&sh.full[warp], phase, abort_flag, wait_limit);
        if (!__all_sync(0xffffffffu, ok)) break;
        phase ^= 1;
        const int k0 = s % parts * ks, kbs = min(ks, in_dim - k0) / 32;     // an even number
        const unsigned char* wrow = ring + (warp * 8 + g) * GT_ROW + kq * 16;
        const uint16_t* xs = xrow + k0;
        float c[4][4] = {};
        auto block = [&](int kb, int u) {
            const uint4 w = *reinterpret_cast<const uint4*>(wrow + kb * 64);
            uint4 a = *reinterpret_cast<const uint4*>(xs + kb * 32);
            if (FORM == GT_SHORT && !live) a = make_uint4(0, 0, 0, 0);
            mma_bf16_16816(c[2 * u], a.x, 0u, a.y, 0u, w.x, w.y);
            mma_bf16_16816(c[2 * u + 1], a.z, 0u, a.w, 0u, w.z, w.w);
        };
        if (FORM == GT_SHORT) {
#pragma unroll 2
            for (int kb = 0; kb < kbs; kb += 2) { block(kb, 0); block(kb + 1, 1); }
        } else if (FORM == GT_WHOLE || kbs == GT_KB) {
#pragma unroll
            for (int kb = 0; kb < GT_KB; ++kb) block(kb, kb & 1);
        } else {
#pragma unroll 1
            for (int kb = 0; kb < kbs; kb += 2) { block(kb, 0); block(kb + 1, 1); }
        }
        __syncwarp();
        fence_proxy_async();                                                // the slot's reads before the copy that refills it
        fetch(s + 2 * GT_WARPS);
        put(s, c);
    }
    __syncthreads();
    if (sh.abort_flag) {
        // Somebody gave up.  Copies already issued still land in this block's shared memory: give every barrier a
        // bounded chance to complete before the memory is released.
        if (threadIdx.x == 0) {
            for (int i = 0; i < GT_SLOTS; ++i)
                for (unsigned p = 0; p < 2; ++p)
                    for (unsigned w = 0; w < (1u << 12) && !mbar_test(&sh.full[i], p); ++w) __nanosleep(32);
            atomicCAS(&ctrl->status, 0, -5);   // SVLM_ERR_TIMEOUT
        }
        __syncthreads();
        return;
    }
    for (int i = threadIdx.x; i < (r1 - r0) * n; i += GT_WARPS * 32) {
        const int t = i / (r1 - r0), r = i - t * (r1 - r0);
        float sum = 0.f;
        for (int p = 0; p < parts; ++p) sum += sh.part[(r >> 3) * parts + p][t][r & 7];
        Y[(size_t)t * out_dim + r0 + r] = __bfloat16_as_ushort(__float2bfloat16_rn(sum));
    }
}

// Elements of K per stage: as few stages as go, about equally long, all but the last a multiple of 64.
int few_stage(int in_dim) {
    const int parts = (in_dim + GT_KS - 1) / GT_KS;
    return ((in_dim + parts - 1) / parts + 63) / 64 * 64;
}

template <int FORM>
cudaError_t launch_few(const uint16_t* X, const uint16_t* W, uint16_t* Y, int n, int in_dim, int out_dim, SvlmCtrl* ctrl, cudaStream_t st) {
    const size_t fixed = (size_t)GT_SLOTS * 8 * GT_ROW + sizeof(GtShared);
    // (the limit of the longest token rows this kernel takes, so that a later call finds it raised)
    const cudaError_t e = svlm_allow_smem<gemv_few_kernel<FORM>>(fixed + GT_MAX_X);
    if (e != cudaSuccess) return e;
    const int parts = (in_dim + GT_KS - 1) / GT_KS, ks = few_stage(in_dim);
    const int most_rows = GT_MAX_STAGES / parts * 8;
    const int blocks = std::max(std::min((out_dim + 7) / 8, svlm_sm_count()), (out_dim + most_rows - 1) / most_rows);
    return svlm_launch_chained(gemv_few_kernel<FORM>, dim3(blocks), dim3(GT_WARPS * 32), fixed + (size_t)n * (in_dim + GT_PAD) * 2, 1, st, X, W, Y, n,
                               in_dim, out_dim, parts, ks, ctrl);
}

// What the kernel above takes: the token rows fit beside the ring, a group's stages fit the partial sums, and the last
// stage of a group is not empty (in_dim is a multiple of 64).
bool few_supported(int n, int in_dim) {
    const int parts = (in_dim + GT_KS - 1) / GT_KS, ks = few_stage(in_dim);
    return n <= 4 && in_dim % 64 == 0 && parts <= GT_MAX_STAGES && (parts - 1) * ks < in_dim && (size_t)n * (in_dim + GT_PAD) * 2 <= GT_MAX_X;
}

// More tokens, up to 16 (or longer rows than the kernel above takes): the tokens are the M = 16 rows of mma.sync.m16n8k16, eight rows of W the N.  A block owns
// eight output rows; its eight warps split K (k-blocks of 32, strided), every lane loading 16 bytes of one W
// row and of two token rows per k-block straight into the fragment registers (the dot product does not care
// in which order k is summed, so the eight consecutive elements a lane loads serve two MMAs), several k-blocks
// in flight; the warps' partial tiles meet in shared memory.
constexpr int GM_KB_IN_FLIGHT = 7;

__global__ void __launch_bounds__(GV_THREADS, 4) gemv_mma_kernel(const uint16_t* X, const uint16_t* __restrict__ W,
                                                             uint16_t* __restrict__ Y, int n, int in_dim, int out_dim) {
    __shared__ float part[GV_THREADS / 32][16][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, kq = lane & 3;
    const int row0 = blockIdx.x * 8;
    const int wrow = min(row0 + g, out_dim - 1);
    const uint4* wp = reinterpret_cast<const uint4*>(W + (size_t)wrow * in_dim) + kq;          // + 4 per k-block of 32
    const uint4* xlo = reinterpret_cast<const uint4*>(X + (size_t)min(g, n - 1) * in_dim) + kq;
    const uint4* xhi = reinterpret_cast<const uint4*>(X + (size_t)min(g + 8, n - 1) * in_dim) + kq;
    const bool lo_live = g < n, hi_live = g + 8 < n;
    const int n_kb = in_dim / 32;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    uint4 w[GM_KB_IN_FLIGHT];
    auto load_w = [&](int kb0) {
#pragma unroll
        for (int u = 0; u < GM_KB_IN_FLIGHT; ++u) {
            const int kb = kb0 + u * (GV_THREADS / 32);
            w[u] = kb < n_kb ? __ldg(wp + 4 * kb) : make_uint4(0, 0, 0, 0);
        }
    };
    // as above: the first batch of weights is fetched before the wait for the predecessor, the rest asked into L2
    // (5 tokens, 33 MB: 8.75 -> 7.7 us)
    svlm_ptx::pdl_launch_dependents();
    load_w(warp);
    for (int kb = warp + (GV_THREADS / 32) * GM_KB_IN_FLIGHT; kb < n_kb; kb += GV_THREADS / 32)
        if ((kb & 1) == 0 && kq == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(wp + 4 * kb));
    svlm_ptx::pdl_wait();
    for (int kb0 = warp; kb0 < n_kb; kb0 += (GV_THREADS / 32) * GM_KB_IN_FLIGHT) {
        uint4 a[GM_KB_IN_FLIGHT], bq[GM_KB_IN_FLIGHT];
        if (kb0 != warp) load_w(kb0);
#pragma unroll
        for (int u = 0; u < GM_KB_IN_FLIGHT; ++u) {
            const int kb = kb0 + u * (GV_THREADS / 32);
            const bool live = kb < n_kb;
            a[u] = live && lo_live ? svlm_ptx::ld_in(xlo + 4 * kb) : make_uint4(0, 0, 0, 0);
            bq[u] = live && hi_live ? svlm_ptx::ld_in(xhi + 4 * kb) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < GM_KB_IN_FLIGHT; ++u) {
            mma_bf16_16816(c, a[u].x, bq[u].x, a[u].y, bq[u].y, w[u].x, w[u].y);
            mma_bf16_16816(c, a[u].z, bq[u].z, a[u].w, bq[u].w, w[u].z, w[u].w);
        }
    }
    part[warp][g][2 * kq] = c[0];
    part[warp][g][2 * kq + 1] = c[1];
    part[warp][g + 8][2 * kq] = c[2];
    part[warp][g + 8][2 * kq + 1] = c[3];
    __syncthreads();
    if (threadIdx.x < 128) {
        const int t = threadIdx.x >> 3, r = threadIdx.x & 7;
        float s = 0.f;
#pragma unroll
        for (int w8 = 0; w8 < GV_THREADS / 32; ++w8) s += part[w8][t][r];
        if (t < n && row0 + r < out_dim) Y[(size_t)t * out_dim + row0 + r] = __bfloat16_as_ushort(__float2bfloat16_rn(s));
    }
}

}  // namespace

bool svlm_gemv_supported(int n, int in_dim) { return n >= 1 && n <= 16 && in_dim % 32 == 0 && (size_t)4 * in_dim * 2 <= 200 * 1024; }

cudaError_t svlm_launch_gemv(const void* X, const void* W, void* Y, int n, int in_dim, int out_dim, bool from_l2, SvlmCtrl* ctrl, cudaStream_t st) {
    const uint16_t* x = static_cast<const uint16_t*>(X);
    const uint16_t* w = static_cast<const uint16_t*>(W);
    uint16_t* y = static_cast<uint16_t*>(Y);
    // Weights that stay in L2 from token to token: fetching ahead buys nothing, and more, smaller blocks are faster while a warp
    // of theirs has all its weights in flight at once (rows of up to 1792), or in two batches and there are two blocks per SM:
    // us, one and four tokens, this kernel against the other: 1024 x 1536 2.28 and 2.46 / 2.13 and 2.36, 1344 x 4096 2.57 and 2.60 / 2.94
    // and 3.54, 1792 x 2048 2.56 and 2.62 / 2.47 and 2.99, 2560 x 4096 4.65 and 4.61 / 4.61 and 4.81, 3584 x 2560 4.77 and 5.03 / 4.56 and
    // 5.25, 3584 x 4608 5.33 and 5.47 / 5.92 and 6.66.  Not with fewer rows of W (3584 x 2048 4.47 and 4.66 / 3.44 and 4.05, x 512 3.72 and
    // 3.81 / 2.53 and 3.23), longer ones (4096 x 1536 6.16 and 6.39 / 3.54 and 3.71, 8192 x 1024 7.95 and 8.24 / 3.80 and 4.48) or such as lie a multiple of
    // 4 KB apart (2048 x 6144 6.50 and 6.69 / 4.66 and 4.74).
    const bool in_batches = in_dim <= 1792 || (in_dim <= 3584 && in_dim % 2048 && out_dim / 8 >= 2 * svlm_sm_count());
    if (few_supported(n, in_dim) && !(from_l2 && in_batches)) {
        const auto launch = in_dim % GT_KS == 0 ? launch_few<GT_WHOLE> : few_stage(in_dim) == GT_KS ? launch_few<GT_MIXED> : launch_few<GT_SHORT>;
        return launch(x, w, y, n, in_dim, out_dim, ctrl, st);
    }
    return svlm_launch_chained(gemv_mma_kernel, dim3((out_dim + 7) / 8), dim3(GV_THREADS), 0, 1, st, x, w, y, n, in_dim, out_dim);
}
