// Q/K/V projection whose epilogue appends to the cache (sm_100a): the step on the input side of the
// per-chunk path.  For the n new tokens of a layer, Y = X W^T with W = [W_q; W_k; W_v]; the query columns
// go to the caller's Q buffer, the key columns are rotated at each token's contiguous position
// (paper Section 2.1, "Contiguous RoPE") and written, with the value columns, straight into the
// token's cache slot: K and V never make a round trip through global memory between the GEMM and
// the cache.  The plain projection after the attention is the same kernel.
//
// A dense contraction, so it runs on the tensor cores.  Two CTAs work as a pair (cta_group::2) on a tile of 256 output
// features x N tokens, each bringing in its own 128 rows of W and half of the tokens' rows.  The features are the M side:
// with tokens there, a chunk of 524 would fill 3 tiles of 256 (a third of it padding); as the N side they are cut in equal
// tiles of any multiple of 32, and the launch picks the width that fills the SM pairs best (svlm_proj_tile).
// What bounded the kernel was the pace of its single threads, not memory or math: 690 cycles per k-block in the issuing
// thread (stage numbers by division, descriptors moved into uniform registers one by one), whatever the tile, so that 32
// to 1024 tokens all took 25-29 us at hidden 3584.  With counted stages, the whole warp in the issuer's loop and two
// producers a k-block takes the 2 N cycles of its math, from N = 160 on; below that the issuer's 320.
// Hidden 3584, 4608 features, us: 32 tokens 25.4 -> 12.5, 531 tokens 27.6 -> 17.1, 1024 tokens 29.2 -> 25.3, 4096 tokens
// 107 -> 99 (1364 TFLOP/s; the clock then drops with the power limit).
//   warps 0, 10  TMA (128-byte swizzle) into a ring of up to eight stages, in turns; both CTAs' bytes are counted on the
//                leader's barrier
//   warp 1       of the leading CTA: one thread issues tcgen05.mma M256 N K16 into N TMEM columns of both CTAs
//   warps 2-9    epilogue: a CTA's 128 accumulator rows are one head; they are transposed through shared memory (the ring,
//                idle by then), so that a token's row leaves in one coalesced 256-byte store and a key's rotation
//                partners j, j + 64 meet in one lane
// Every mbarrier wait is bounded; on expiry the CTA records SVLM_ERR_TIMEOUT, drains its copies, meets its partner at the
// cluster barrier, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_ptx.cuh"
#include "svlm_rope.cuh"
#include "svlm_tc.cuh"

namespace {

using namespace svlm_ptx;
using namespace svlm_tc;

constexpr int QK_MAX_STAGES = 8;
constexpr int QK_RING = 6 * 32768;              // bytes: six stages of the widest tile
constexpr int QK_BK = 64;                       // k-block: 64 bf16 = one 128-byte swizzle row
constexpr int QK_W_TILE = 128 * QK_BK * 2;      // bytes of this CTA's rows of W in a stage
constexpr int QK_EPI_WARPS = 8;
constexpr int QK_THREADS = 96 + 32 * QK_EPI_WARPS;   // two producers, the issuer, the epilogue
constexpr int QK_EARLY = 20;                    // tokens per warp whose factors are looked up ahead (a width of 160)
constexpr int QK_EPI_ROW = 128 + 4;             // floats between the transposed rows (16-byte aligned, conflict-free)
static_assert(256 * QK_EPI_ROW * 4 <= QK_RING, "the transposed tile lives in the ring");

struct QkShared {
    unsigned long long full[QK_MAX_STAGES], empty[QK_MAX_STAGES], acc_full;
    unsigned tmem_base;
    int abort_flag;
};

// ---- the paired forms (cta_group::2) ---------------------------------------------------------------------------
// A tile into this CTA's shared memory; the bytes are counted on `bar`, an address of the pair's leading CTA.
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const void* tmap, int x, int y, unsigned bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(bar) : "memory");
}
// The same with an L2 policy.  The weights are marked as read once (l2_read_once): their 59 MB per layer of the 7B shape used to push
// everything else out of L2, the kernels' code included, whose first page then took the chunk prefill 7100 cycles, not 3400.
// 531 tokens with their projections, 28 layers, in a loop at the power limit, both policies on the present code: 3429 -> 3329 us.
// (Projections behind one another with nothing between them only pay for it: 524 tokens 19.95 -> 20.15 us with the append.)
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const void* tmap, int x, int y, unsigned bar, unsigned long long policy) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;"
                 ::"r"(smem_u32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(bar), "l"(policy) : "memory");
}
// D (both CTAs' tensor memory) (+)= A B, operands in both CTAs' shared memory at the same addresses
__device__ __forceinline__ void tc_mma_ss_pair(unsigned d_tmem, unsigned long long a_desc, unsigned long long b_desc, unsigned idesc,
                                               unsigned accumulate) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives on this barrier of both CTAs when the MMAs issued so far have completed.
__device__ __forceinline__ void tc_commit_pair(void* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}

// kv_heads_used = cd.kv_heads for the projection with append; 0 turns the kernel into the plain projection
// Y = X W^T (the output projection after attention): every 128-column block is then a "query head" and goes to Q_out.
// Grid: (2 * pairs of heads, token tiles of `width`), clusters of two.  W_ONCE: the weights are marked as read once; an instance each, since
// an ordinary policy as an operand of the load is not free either (4096 tokens 106.6 us with the append, without 106.3).
template <bool W_ONCE>
__global__ void __launch_bounds__(QK_THREADS, 1)
qkv_append_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ SvlmCacheDev cd,
                  int layer, int n, int hidden, int q_heads, int kv_heads_used, int width, uint16_t* __restrict__ Q_out) {
    constexpr int D = 128, HALF = 64;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring = smem_raw;                                      // [stage][W tile | half of the X tile]
    QkShared& sh = *reinterpret_cast<QkShared*>(ring + QK_RING);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned rank = cluster_rank();
    const int head = blockIdx.x;                 // this CTA's head, in the order query heads, key heads, value heads
    const int n_heads = q_heads + 2 * kv_heads_used;
    const int i0 = blockIdx.y * width;           // first token of the tile
    const int n_kb = hidden / QK_BK;
    const int stage_bytes = QK_W_TILE + width / 2 * 128;
    const int n_stages = min(QK_MAX_STAGES, QK_RING / stage_bytes);
    volatile int* abort_flag = &sh.abort_flag;
    const unsigned wait_limit = ld_l2(&cd.ctrl->wait_limit);   // written at creation only, never by a kernel

    if (smem_u32(smem_raw) & 1023) {             // swizzled tiles need a 1024-byte aligned base; same in every CTA
        if (threadIdx.x == 0) atomicCAS(&cd.ctrl->status, 0, -4);   // SVLM_ERR_CUDA
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < QK_MAX_STAGES; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
        mbar_init(&sh.acc_full, 1);
        sh.abort_flag = 0;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)), "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    // Set up while the predecessor ends (programmatic dependent launch); the wait comes before the trigger.
    pdl_wait();
    pdl_launch_dependents();
    tc_fence_before();
    cluster_sync_all();                          // both CTAs' barriers are initialised
    tc_fence_after();
    const unsigned tmem = sh.tmem_base;

    if (warp == 0 || warp == 2 + QK_EPI_WARPS) {
        // ================= TMA producers, a k-block each in turn =================
        // (this loop and the issuer's are paced by their own instructions, one dependent after the other: stage numbers
        // and phases are counted, not divided out, and addresses advance with them)
        if (lane == 0) {
            const int first = warp ? 1 : 0, y = i0 + (int)rank * (width / 2);
            const unsigned long long once = W_ONCE ? l2_read_once() : 0;
            unsigned bar = map_to_rank(&sh.full[first], 0);
            int st = first;
            unsigned phase = 1;                                  // first pass: already free
            unsigned char* dst = ring + first * stage_bytes;
            for (int kb = first, x = first * QK_BK; kb < n_kb; kb += 2, x += 2 * QK_BK) {
                if (!mbar_wait(&sh.empty[st], phase, abort_flag, wait_limit)) break;
                if (rank == 0) mbar_expect_tx(&sh.full[st], 2 * stage_bytes);
                if (W_ONCE) tma_load_2d_pair(dst, &tmW, x, head * D, bar, once);   // rows past the end read as zeros
                else tma_load_2d_pair(dst, &tmW, x, head * D, bar);
                tma_load_2d_pair(dst + QK_W_TILE, &tmX, x, y, bar);
                dst += 2 * stage_bytes;
                bar += 16;
                if ((st += 2) >= n_stages) { st -= n_stages; phase ^= 1; dst -= n_stages * stage_bytes; bar -= 8 * n_stages; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer (leading CTA) =================
        // The whole warp runs the loop, so that descriptors live in uniform registers; one elected lane executes the
        // tcgen05 instructions.
        if (rank == 0) {
            const bool leader = elect_one();
            const unsigned idesc = make_idesc(256, 0, 0) | ((unsigned)(width >> 3) << 17);
            const unsigned td = __shfl_sync(0xffffffffu, tmem, 0);
            unsigned long long da = smem_desc(smem_u32(ring), 16, 1024), db = smem_desc(smem_u32(ring + QK_W_TILE), 16, 1024);
            const unsigned step = (unsigned)stage_bytes >> 4;
            int st = 0;
            unsigned phase = 0;
            bool ok = true;
            for (int kb = 0; kb < n_kb; ++kb) {
                ok = mbar_wait(&sh.full[st], phase, abort_flag, wait_limit);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < QK_BK / 16; ++ks)
                        tc_mma_ss_pair(td, da + (unsigned)(ks * 32 >> 4), db + (unsigned)(ks * 32 >> 4), idesc, (kb | ks) != 0);
                    tc_commit_pair(&sh.empty[st]);
                }
                __syncwarp();
                da += step;
                db += step;
                if (++st == n_stages) { st = 0; phase ^= 1; da -= (unsigned long long)step * n_stages; db -= (unsigned long long)step * n_stages; }
            }
            if (ok && leader) tc_commit_pair(&sh.acc_full);
        }
        __syncwarp();
    } else {
        // ================= epilogue: this CTA's head, `width` tokens =================
        const int ew = warp - 2, quad = warp & 3;                // quad: the TMEM lane quadrant this warp may read
        const int kv = head - q_heads;                           // < 0: query head; < kv_heads: key head; else value head
        const bool key = kv >= 0 && kv < kv_heads_used;
        // where this warp's tokens (ew, ew + 8, ...; one per lane) live, and their positions, if the append stood
        int slot = -1, c0 = 0, c1 = 0, c2 = 0;
        if (kv >= 0 && head < n_heads) {
            const int t = ew + QK_EPI_WARPS * lane, i = i0 + t;
            if (t < width && i < n && ld_l2(&cd.ctrl->append_n) == n) {
                const int s = ld_l2(cd.new_slot + i);
                if (ld_l2(cd.slot_gid + s) == ld_l2(&cd.ctrl->n_total) - n + i) slot = s;
                if (key) {
                    c0 = ld_l2(cd.slot_c + s);
                    c1 = ld_l2(cd.slot_c + cd.n_slots + s);
                    c2 = ld_l2(cd.slot_c + 2 * (size_t)cd.n_slots + s);
                }
            }
        }
        // A key head: the rotation factors of the warp's first tokens are looked up now, while the tensor pipe is still busy
        // with the tile.  Looked up afterwards they kept the key heads' CTAs behind all others: 23.1 us per call at 292
        // tokens of 3584 features into 28 + 4 + 4 heads, 17.9 now, which is the plain projection's time.
        const int a0 = cd.rope_mode == 0 ? 0 : (2 * lane < cd.sec_t ? 0 : (2 * lane < cd.sec_th ? 1 : 2));
        const int a1 = cd.rope_mode == 0 ? 0 : (2 * lane + 1 < cd.sec_t ? 0 : (2 * lane + 1 < cd.sec_th ? 1 : 2));
        const float2* tab = reinterpret_cast<const float2*>(cd.rope_tab);
        auto factors = [&](int j, float2& f0, float2& f1) {      // of the warp's token j, for pairs 2 lane and 2 lane + 1
            const int p0 = __shfl_sync(0xffffffffu, c0, j), p1 = __shfl_sync(0xffffffffu, c1, j), p2 = __shfl_sync(0xffffffffu, c2, j);
            f0 = svlm_rope_cs_batched(tab, HALF, 2 * lane, a0 == 0 ? p0 : (a0 == 1 ? p1 : p2));
            f1 = svlm_rope_cs_batched(tab, HALF, 2 * lane + 1, a1 == 0 ? p0 : (a1 == 1 ? p1 : p2));
        };
        float2 e0[QK_EARLY], e1[QK_EARLY];
        const int lim = 1 << 16;
        const bool far = __any_sync(0xffffffffu, c0 <= -lim || c0 >= lim || c1 <= -lim || c1 >= lim || c2 <= -lim || c2 >= lim);
        if (key) {
#pragma unroll
            for (int j = 0; j < QK_EARLY; ++j) factors(j, e0[j], e1[j]);
        }
        bool ok = mbar_wait(&sh.acc_full, 0, abort_flag, wait_limit);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
        if (ok) {
            float* tr = reinterpret_cast<float*>(ring) + quad * 32 + lane;
            const unsigned tacc = tmem + ((unsigned)(quad * 32) << 16);
            for (int c32 = ew >> 2; c32 < width / 32; c32 += 2) {
                float v[32];
                tmem_ld32(tacc + c32 * 32, v);
                tmem_wait_ld<32>(v);
#pragma unroll
                for (int k = 0; k < 32; ++k) tr[(c32 * 32 + k) * QK_EPI_ROW] = v[k];
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * QK_EPI_WARPS) : "memory");
        if (ok && head < n_heads) {
            const int here = min(width, n - i0);                 // tokens of the tile
            if (key) {
                uint16_t* k_base = cd.K + ((size_t)layer * cd.kv_heads + kv) * cd.n_slots * D + 2 * lane;
                // pairs (2 lane, 2 lane + 1) with their partners 64 further on, rotated at the slot's current position
                auto put_key = [&](int t, int s, float2 f0, float2 f1) {
                    const float* row = reinterpret_cast<const float*>(ring) + t * QK_EPI_ROW;
                    const float2 x = *reinterpret_cast<const float2*>(row + 2 * lane), y = *reinterpret_cast<const float2*>(row + HALF + 2 * lane);
                    uint16_t* dst = k_base + (size_t)s * D;
                    *reinterpret_cast<unsigned*>(dst) = pack2(x.x * f0.x - y.x * f0.y, x.y * f1.x - y.y * f1.y);
                    *reinterpret_cast<unsigned*>(dst + HALF) = pack2(y.x * f0.x + x.x * f0.y, y.y * f1.x + x.y * f1.y);
                };
                if (!far) {
#pragma unroll
                    for (int j = 0; j < QK_EARLY; ++j) {
                        const int s = __shfl_sync(0xffffffffu, slot, j), t = ew + QK_EPI_WARPS * j;
                        if (t < here && s >= 0) put_key(t, s, e0[j], e1[j]);
                    }
                }
#pragma unroll 4
                for (int j = far ? 0 : QK_EARLY; j < 32; ++j) {
                    const int t = ew + QK_EPI_WARPS * j;
                    if (t >= here) break;
                    const int s = __shfl_sync(0xffffffffu, slot, j);
                    float2 f0, f1;
                    factors(j, f0, f1);
                    if (far) {                                   // native positions of a long stream
                        const int p0 = __shfl_sync(0xffffffffu, c0, j), p1 = __shfl_sync(0xffffffffu, c1, j), p2 = __shfl_sync(0xffffffffu, c2, j);
                        f0 = svlm_rope_cs(tab, HALF, 2 * lane, a0 == 0 ? p0 : (a0 == 1 ? p1 : p2), cd.theta[2 * lane]);
                        f1 = svlm_rope_cs(tab, HALF, 2 * lane + 1, a1 == 0 ? p0 : (a1 == 1 ? p1 : p2), cd.theta[2 * lane + 1]);
                    }
                    if (s >= 0) put_key(t, s, f0, f1);
                }
            } else {
                // query head -> the caller's buffer; value head -> the cache slot: a plain bf16 copy of the row, two rows
                // at a time (half a warp each)
                const int sub = lane >> 4, e = (lane & 15) * 8;
                uint16_t* q_base = Q_out + ((size_t)i0 * q_heads + head) * D + e;
                uint16_t* v_base = cd.V + ((size_t)layer * cd.kv_heads + (kv - kv_heads_used)) * cd.n_slots * D + e;
#pragma unroll 4
                for (int j = 0; j < 32; j += 2) {
                    const int t = ew + QK_EPI_WARPS * (j + sub);
                    if (ew + QK_EPI_WARPS * j >= here) break;
                    const int s = __shfl_sync(0xffffffffu, slot, j + sub);
                    if (t >= here || (kv >= 0 && s < 0)) continue;
                    const float* row = reinterpret_cast<const float*>(ring) + t * QK_EPI_ROW + e;
                    const float4 x = *reinterpret_cast<const float4*>(row), y = *reinterpret_cast<const float4*>(row + 4);
                    uint16_t* dst = kv < 0 ? q_base + (size_t)t * q_heads * D : v_base + (size_t)s * D;
                    *reinterpret_cast<uint4*>(dst) = make_uint4(pack2(x.x, x.y), pack2(x.z, x.w), pack2(y.x, y.y), pack2(y.z, y.w));
                }
            }
        }
    }

    // ---- teardown ------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (sh.abort_flag && threadIdx.x == 0) {   // copies already issued still land here: give every stage a bounded chance to complete
        for (int s = 0; s < QK_MAX_STAGES; ++s)
            for (unsigned p = 0; p < 2; ++p)
                for (unsigned w = 0; w < (1u << 16) && !mbar_test(&sh.full[s], p); ++w) __nanosleep(32);
        atomicCAS(&cd.ctrl->status, 0, -5);   // SVLM_ERR_TIMEOUT
    }
    __syncthreads();
    cluster_sync_all();                          // neither CTA's memory is read or signalled by the other's work any more
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
    }
}

constexpr size_t qkv_smem() { return (size_t)QK_RING + sizeof(QkShared); }

}  // namespace

// Tokens per tile: the width at which the rounds of SM pairs, each as long as its math (2 N cycles per k-block, or the 320
// that the issuer needs) and 14,000 cycles for filling the pipe and the epilogue, end first.
int svlm_proj_tile(int n, int hidden, int blocks128) {
    const int pairs_sm = std::max(1, svlm_sm_count() / 2), tiles_m = (blocks128 + 1) / 2;
    int best = 256;
    long long best_cost = -1;
    for (int w = 32; w <= 256; w += 32) {
        const long long tiles = (long long)tiles_m * ((n + w - 1) / w);
        const long long rounds = (tiles + pairs_sm - 1) / pairs_sm;
        const long long cost = rounds * ((long long)std::max(2 * w, 320) * (hidden / QK_BK) + 14000);
        if (best_cost < 0 || cost <= best_cost) { best_cost = cost; best = w; }
    }
    return best;
}

cudaError_t svlm_launch_qkv_append(const void* tmX, const void* tmW, const SvlmCacheDev& cd, int layer, int n, int hidden,
                                   int q_heads, bool with_append, int width, void* Q_out, cudaStream_t st) {
    const int kv = with_append ? cd.kv_heads : 0;
    const dim3 grid((q_heads + 2 * kv + 1) / 2 * 2, (n + width - 1) / width);
    // Read once: all tiles at a time, so that whoever shares rows of W reads them together and nobody later (4133 tokens, where later tiles
    // read them again: 2103 us with an ordinary policy, 2149 as read once); and not where all layers' weights, on both sides of the
    // attention and taken to be of this one's size, stay in L2 from pass to pass and a short chunk leaves them there.  Chunk with both
    // projections, us a layer, ordinary policy and read once: hidden 1024, four layers, 20 tokens 30.05 and 30.48, 133 tokens 35.07 and 35.21, 524
    // 58.18 and 57.78; hidden 2048, three layers (57 MB), 20 tokens 35.95 and 36.40, 524 57.1 and 56.1, four layers, 133 tokens 43.65 and 43.17;
    // hidden 3584, one layer (59 MB), 20 tokens 56.6 and 57.4, 133 74.8 and 75.9, 200 78.9 and 75.7, 524 84.1 and 78.8, two layers, 20 tokens 53.6 and 51.4.
    const size_t all = (size_t)cd.layers * 2 * grid.x * 128 * hidden * 2;
    const bool w_once = (int)(grid.x * grid.y) <= svlm_sm_count() && (n >= 160 || all >= (size_t)64 << 20);
    const auto launch = [&](auto once) {
        constexpr auto kernel = qkv_append_kernel<decltype(once)::value>;
        const cudaError_t e = svlm_allow_smem<kernel>(qkv_smem());
        if (e != cudaSuccess) return e;
        return svlm_launch_chained(kernel, grid, dim3(QK_THREADS), qkv_smem(), 2, st, *static_cast<const CUtensorMap*>(tmX),
                                   *static_cast<const CUtensorMap*>(tmW), cd, layer, n, hidden, q_heads, kv, width, static_cast<uint16_t*>(Q_out));
    };
    return w_once ? launch(std::true_type{}) : launch(std::false_type{});
}
