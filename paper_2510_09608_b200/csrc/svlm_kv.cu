// Key/value movement: writing appended tokens into their slots with the first rotation, and the
// in-place re-rotation of retained keys after an eviction (paper Section 2.1, "Contiguous RoPE":
// the indices of later tokens are shifted left; a stored key R(c)k becomes R(c-E)k = R(-E)R(c)k).
// Both are streaming kernels: 16-byte accesses, no reuse, bound by HBM bandwidth.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include "svlm_dev.h"
#include "svlm_launch.h"
#include "svlm_ptx.cuh"
#include "svlm_rope.cuh"
#include "svlm_rotate.cuh"

namespace {

// One thread per (token, group of 8 pairs) and per share of the [layer][kv_head] rows (blockIdx.y), so the rotation
// factors are looked up once per share (table, see svlm_rope.cuh).  What bounds it is latency: source rows, and the chain
// new slot -> position -> factors, which depend on nothing of each other.  early != 0: the caller vouches that no kernel
// that may still be running writes this cache's metadata; the chain is then walked before the wait for the predecessor
// (programmatic dependent launch), which leaves one round trip to memory after it.  Per layer of a 524-token chunk
// between two chunk-prefill launches: 8.3 us in the stream with 17 blocks, a longer chain and a full launch gap, then 4.3.
// The successor is let start behind the wait in either case: kernels that do nothing but wait, load and store follow one another in
// 2.1 us that way and in 2.8 to 3.4 if each starts the next one first (68 and 148 blocks; 2.0 to 4.1 for plain launches).
// Eight streams' writes a layer, chunk of 28 layers: 15,087 -> 14,964 us, one stream 2258 -> 2242.
template <int UNROLL>
__global__ void __launch_bounds__(256) kv_write_kernel(SvlmCacheDev cd, int layer, const uint16_t* K,
                                                       const uint16_t* V, int n, int rows_per_block, int early) {
    if (!early) {
        svlm_ptx::pdl_wait();
        svlm_ptx::pdl_launch_dependents();
    }
    const int half = cd.head_dim / 2;
    const int gshift = cd.head_dim == 128 ? 3 : 2;      // log2 of the groups (threads) per token
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = t >> gshift, g = t & ((1 << gshift) - 1);
    const bool live = i < n;
    const int d = cd.head_dim;
    const int n_rows = layer < 0 ? cd.layers * cd.kv_heads : cd.kv_heads;      // rows of [layer][kv_head] in this call
    const int row0 = blockIdx.y * rows_per_block, row1 = min(n_rows, row0 + rows_per_block);
    const int first_row = layer < 0 ? 0 : layer * cd.kv_heads;                 // of the cache
    // source of row r: [layer (only when all layers are given)][token][kv_head]
    auto src_of = [&](int r) {
        const int l = r / cd.kv_heads, h = r - l * cd.kv_heads;
        return (((size_t)l * n + i) * cd.kv_heads + h) * d + g * 8;
    };
    Bf16x8 lo[UNROLL], hi[UNROLL];
    uint4 vlo[UNROLL], vhi[UNROLL];
    auto load_rows = [&](int r) {
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (live && r + u < row1) {
                const size_t src = src_of(r + u);
                lo[u] = bf16x8(svlm_ptx::ld_in(reinterpret_cast<const uint4*>(K + src)));
                hi[u] = bf16x8(svlm_ptx::ld_in(reinterpret_cast<const uint4*>(K + src + half)));
                vlo[u] = svlm_ptx::ld_in(reinterpret_cast<const uint4*>(V + src));
                vhi[u] = svlm_ptx::ld_in(reinterpret_cast<const uint4*>(V + src + half));
            }
    };
    if (!early) load_rows(row0);
    const int append_n = svlm_ptx::ld_l2(&cd.ctrl->append_n);
    const long long n_total = svlm_ptx::ld_l2(&cd.ctrl->n_total);
    int slot = live ? svlm_ptx::ld_l2(cd.new_slot + i) : -1;      // (of an append that was dropped: left over, not used)
    float cs[8], sn[8];
    if (slot >= 0) {
        // A layer's keys may arrive after an eviction has already shifted these tokens (layers are
        // computed one after another): rotate at the slot's CURRENT position, and skip a token that
        // the eviction has dropped in the meantime.
        const long long gid = svlm_ptx::ld_l2(cd.slot_gid + slot);
        int c[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) c[k] = svlm_ptx::ld_l2(cd.slot_c + (size_t)k * cd.n_slots + slot);
        first_rotation(cd, g, c, cs, sn);
        if (gid != n_total - n + i) slot = -1;
    }
    if (early) {
        svlm_ptx::pdl_wait();
        svlm_ptx::pdl_launch_dependents();
        load_rows(row0);
    }
    if (append_n != n || slot < 0) return;   // the metadata append was dropped (capacity) or does not match
    for (int r = row0; r < row1; r += UNROLL) {
        if (r != row0) load_rows(r);
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (r + u < row1) {
                const size_t dst = ((size_t)(first_row + r + u) * cd.n_slots + slot) * d + g * 8;
                rotate8(lo[u], hi[u], cs, sn);
                *reinterpret_cast<Bf16x8*>(cd.K + dst) = lo[u];
                *reinterpret_cast<Bf16x8*>(cd.K + dst + half) = hi[u];
                *reinterpret_cast<uint4*>(cd.V + dst) = vlo[u];
                *reinterpret_cast<uint4*>(cd.V + dst + half) = vhi[u];
            }
    }
}

// Re-rotation after an eviction.  grid.x covers the slots, grid.y splits the layers.  A thread owns
// (slot, group of 8 pairs) and walks its share of the [layer][kv_head] rows with the same sines;
// the angle -E*theta is identical on the three MRoPE axes because all three indices of a token
// shift by the same E.
template <int UNROLL>
__device__ __forceinline__ void evict_rotate_body(const SvlmCacheDev& cd, int layers_per_block) {
    if (!cd.ctrl->evict_moved) return;
    const int half = cd.head_dim / 2;
    const int groups = half / 8;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int slot = t / groups, g = t % groups;
    if (slot >= cd.n_slots) return;
    const int delta = cd.slot_delta[slot];
    if (delta == 0) return;
    float cs[8], sn[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float2 f = svlm_rope_cs(reinterpret_cast<const float2*>(cd.rope_tab), half, g * 8 + j, -(long long)delta,
                                      cd.theta[g * 8 + j]);
        cs[j] = f.x;
        sn[j] = f.y;
    }
    const int d = cd.head_dim;
    const int row0 = blockIdx.y * layers_per_block * cd.kv_heads;
    const int row1 = min(cd.layers, (blockIdx.y + 1) * layers_per_block) * cd.kv_heads;
    const size_t stride = (size_t)cd.n_slots * d;
    uint16_t* base = cd.K + (size_t)slot * d + g * 8;
    for (int r = row0; r < row1; r += UNROLL) {
        Bf16x8 lo[UNROLL], hi[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (r + u < row1) {
                lo[u] = *reinterpret_cast<const Bf16x8*>(base + (r + u) * stride);
                hi[u] = *reinterpret_cast<const Bf16x8*>(base + (r + u) * stride + half);
            }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (r + u < row1) {
                rotate8(lo[u], hi[u], cs, sn);
                *reinterpret_cast<Bf16x8*>(base + (r + u) * stride) = lo[u];
                *reinterpret_cast<Bf16x8*>(base + (r + u) * stride + half) = hi[u];
            }
    }
}

template <int UNROLL>
__global__ void __launch_bounds__(256) evict_rotate_kernel(SvlmCacheDev cd, int layers_per_block) {
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    evict_rotate_body<UNROLL>(cd, layers_per_block);
}

// Batched form: blockIdx.z selects the cache, whose descriptor is first copied to shared memory.
template <int UNROLL>
__global__ void __launch_bounds__(256) evict_rotate_batch_kernel(SvlmCacheList list, int layers_per_block) {
    __shared__ SvlmCacheDev s_cd;
    svlm_load_desc(&s_cd, list.cd[blockIdx.z]);
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    evict_rotate_body<UNROLL>(s_cd, layers_per_block);
}

// Layers per block in y: enough blocks to fill the machine a few times over, at least 4 rows per thread.
int rotate_layers_per_block(int layers, int kv_heads) {
    int splits = 1;
    while (splits < layers && (layers + splits - 1) / splits * kv_heads > 8) ++splits;
    return (layers + splits - 1) / splits;
}

}  // namespace

cudaError_t svlm_launch_kv_write(const SvlmCacheDev& cd, int layer, const void* K, const void* V, int n, int early, cudaStream_t st) {
    const int threads = n * (cd.head_dim / 16);
    const int x = (threads + 255) / 256;
    const int rows = layer < 0 ? cd.layers * cd.kv_heads : cd.kv_heads;
    // one row per thread while that leaves the grid at a few blocks per SM, then up to eight
    int per = 1;
    while (per < 8 && (long long)x * ((rows + per - 1) / per) > 8 * svlm_sm_count()) per *= 2;
    const dim3 grid(x, (rows + per - 1) / per);
    const uint16_t* k = static_cast<const uint16_t*>(K);
    const uint16_t* v = static_cast<const uint16_t*>(V);
    return per < 4 ? svlm_launch_chained(kv_write_kernel<1>, grid, dim3(256), 0, 1, st, cd, layer, k, v, n, per, early)
                   : svlm_launch_chained(kv_write_kernel<4>, grid, dim3(256), 0, 1, st, cd, layer, k, v, n, per, early);
}

cudaError_t svlm_launch_evict_rotate(const SvlmCacheDev& cd, cudaStream_t st) {
    const int groups = cd.head_dim / 16;
    const int threads = cd.n_slots * groups;
    const int lpb = rotate_layers_per_block(cd.layers, cd.kv_heads);
    dim3 grid((threads + 255) / 256, (cd.layers + lpb - 1) / lpb);
    return svlm_launch_chained(evict_rotate_kernel<4>, grid, dim3(256), 0, 1, st, cd, lpb);
}

cudaError_t svlm_launch_evict_rotate_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, cudaStream_t st) {
    const int threads = geom.n_slots * (geom.head_dim / 16);
    const int lpb = rotate_layers_per_block(geom.layers, geom.kv_heads);
    dim3 grid((threads + 255) / 256, (geom.layers + lpb - 1) / lpb, list.n);
    return svlm_launch_chained(evict_rotate_batch_kernel<4>, grid, dim3(256), 0, 1, st, list, lpb);
}
