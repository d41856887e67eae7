// Host-side launchers of the kernels (one translation unit per kernel family).
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "svlm_dev.h"

void svlm_count_launch();

// Raises a kernel's dynamic shared-memory limit, once per device (the attribute belongs to the device's
// context) and safe to call from several host threads.  The current device is the one the launch goes to.
template <auto Kernel>
cudaError_t svlm_allow_smem(size_t bytes) {
    static std::atomic<unsigned long long> done{0};   // one bit per device, one word per kernel instantiation
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull)) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev, std::memory_order_release);
    return e;
}

// Launches a kernel that may become resident while its predecessor in the stream ends (programmatic dependent launch: the
// kernel itself waits, griddepcontrol), as clusters of `cluster` CTAs, and counts it.
template <typename T>
struct svlm_same { typedef T type; };
template <typename... P>
cudaError_t svlm_launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, int cluster, cudaStream_t st,
                                const typename svlm_same<P>::type&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    svlm_count_launch();
    void* at[] = {const_cast<void*>(static_cast<const void*>(&args))...};      // (kilobytes of parameters: no copies on the way)
    const cudaError_t e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kernel), at);
    if (e != cudaSuccess) cudaGetLastError();      // reported here, not to whoever asks the runtime next
    return e;
}

// Streaming multiprocessors of the current device (looked up once per device).
inline int svlm_sm_count() {
    static std::atomic<int> known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    int n = known[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
        known[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// metadata (svlm_meta.cu).  Where one of these fails, whatever was to follow it must not be launched: it would take the
// metadata of the operation before for its own.
cudaError_t svlm_launch_append_meta(const SvlmCacheDev& cd, const unsigned char* types, const int* pos, int n, cudaStream_t st);
// rotate: the launch re-rotates the moved keys too (svlm_evict_in_one; otherwise svlm_launch_evict_rotate has to follow).
// stored: what the cache is expected to hold (the route depends on it, the result does not)
bool svlm_evict_in_one(const SvlmCacheDev& cd, long long stored);
cudaError_t svlm_launch_evict_meta(const SvlmCacheDev& cd, bool rotate, cudaStream_t st);
// an append's metadata and its keys and values (svlm_launch_kv_write's) in one launch, where svlm_append_in_one says so
bool svlm_append_in_one(const SvlmCacheDev& cd, int layer, int n);
cudaError_t svlm_launch_append_in_one(const SvlmCacheDev& cd, int layer, const void* K, const void* V, const unsigned char* types, const int* pos, int n, cudaStream_t st);
// batched forms, one block per cache: types [n_caches][n], pos [n_caches][n](x3); every cache has the geometry of geom
cudaError_t svlm_launch_append_meta_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, const unsigned char* types, const int* pos, int n,
                                   cudaStream_t st);
cudaError_t svlm_launch_evict_meta_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, bool rotate, cudaStream_t st);

// small transfers from and to page-locked host memory (svlm_host_io.cu); 16-byte aligned, sizes rounded up to 16
cudaError_t svlm_launch_host_in(void* dst, const void* src, size_t bytes, cudaStream_t st);
cudaError_t svlm_launch_host_out(void* dst, const void* src, size_t bytes, unsigned* done, unsigned ticket, cudaStream_t st);

// key/value movement (svlm_kv.cu)
// layer < 0: K,V are [layers][n][kv_heads][d]; otherwise [n][kv_heads][d] for that layer.
// early != 0: the caller vouches that no kernel still running when this one may start writes the cache's metadata.
cudaError_t svlm_launch_kv_write(const SvlmCacheDev& cd, int layer, const void* K, const void* V, int n, int early, cudaStream_t st);
cudaError_t svlm_launch_evict_rotate(const SvlmCacheDev& cd, cudaStream_t st);
// every cache of the list has the geometry of geom
cudaError_t svlm_launch_evict_rotate_batch(const SvlmCacheList& list, const SvlmCacheDev& geom, cudaStream_t st);

// attention (svlm_attend_simple.cu)
// Q, out: [n_caches][n_layers][n_q][q_heads][d]; q_pos: [n_caches][n_q](x3)
void svlm_launch_attend_simple(const SvlmAttendBatch& b, int layer0, int n_layers, const void* Q, const int* q_pos,
                               int n_q, int q_heads, void* out, cudaStream_t st);

// split-KV decode, n_q = 1 (svlm_decode.cu)
size_t svlm_decode_ws_floats(int layers_in_launch, int kv_heads, int head_dim, int splits);
int svlm_decode_splits(int n_pages, int kv_heads, int problems);
// The kernel keeps the list of active pages in shared memory: caches with more pages take the general kernel.
bool svlm_decode_supported(int n_pages);
// Knew/Vnew non-null: fused decode step, the latest appended token's key and value ([caches*layers][kv_heads][d],
// un-rotated) are written to the cache by this launch.  early_loads != 0: the caller vouches that no kernel
// enqueued since the one before the previous launch on this stream wrote this cache's metadata or the pages of the
// layers attended here, so the kernel may read them before the previous kernel has finished.
// early_loads == 2: moreover that previous kernel was itself a decode step of this cache (the per-layer kernel then
// paces its read-ahead, one unit's worth per warp at a time).
// list non-null: the caches have one layer, and the token's metadata is appended by this launch too (types [n_caches],
// positions q_pos); null: svlm_launch_append_meta has run before, or nothing is appended.
// tagged: the per-layer kernel (one layer of one or a few caches; its splits hand their partial results over in tagged
// words in the views' areas of svlm_decode_tagged_bytes, sized for one cache's splits); otherwise the streaming kernel
// with its arrival counters in the views' scratch.
cudaError_t svlm_launch_decode(const SvlmAttendBatch& b, int layer0, int n_layers, const void* Q, const int* q_pos,
                               int q_heads, void* out, int splits, const void* Knew, const void* Vnew, int early_loads,
                               bool tagged, const SvlmCacheList* list, const unsigned char* types, cudaStream_t st);
// Splits of the per-layer kernel for one layer of n_caches caches with `pages` pages or fewer, 0 where the streaming kernel
// is the better one (either gives the same result).
int svlm_decode_layer_splits(int n_pages, int pages, int layers, int kv_heads, int n_caches, int head_dim);
size_t svlm_decode_tagged_bytes(int kv_heads, int head_dim, int splits);

// Q/K/V projection with the append as its epilogue, head_dim 128 (svlm_qkv_sm100.cu).  tmX, tmW: host copies of
// the CUtensorMap of X [n][hidden] (64 x width / 2 box) and W [(q_heads + 2 kv_heads) * 128][hidden] (64 x 128 box), 128-byte
// swizzle; width: svlm_proj_tile for the number of 128-row blocks of W.
// with_append = false: the plain projection Y = X W^T with q_heads blocks of 128 output columns, all written to Q_out.
int svlm_proj_tile(int n, int hidden, int blocks128);
cudaError_t svlm_launch_qkv_append(const void* tmX, const void* tmW, const SvlmCacheDev& cd, int layer, int n, int hidden,
                                   int q_heads, bool with_append, int width, void* Q_out, cudaStream_t st);

// Y = X W^T for a few rows of X (decode-time projections), a bandwidth kernel (svlm_gemv.cu)
bool svlm_gemv_supported(int n, int in_dim);
// from_l2: W is likely to be in L2 already.  ctrl: where a wait that runs out is recorded, and the poll limit
cudaError_t svlm_launch_gemv(const void* X, const void* W, void* Y, int n, int in_dim, int out_dim, bool from_l2, SvlmCtrl* ctrl, cudaStream_t st);

// tcgen05/TMEM/TMA chunk prefill, n_q >= 2 (svlm_prefill_sm100.cu)
bool svlm_prefill_supported(int n_pages, int group);
// counters: svlm_prefill_counter_bytes of the first cache, zero before the first launch (the kernel leaves them zero);
// slots: its svlm_prefill_slot_bytes (0: null).  Launches that share them must not overlap.  held: what each cache is
// expected to hold (the kernel and the balance of the work depend on it, the result only in the order of its sums).
struct SvlmPrefillLoad {
    int pages;      // stored pages
    int windows;    // most tokens the windows keep, i.e. most of a chunk that can be stored
};
// few rows over few pages: a kernel of their own (svlm_prefill_small.cu)
struct SvlmPrefillSmall {
    int tiles;      // of 16 rows per CTA; 0: the tensor-core kernel's business
    int parts;      // CTAs (a cluster) that divide the keys
};
SvlmPrefillSmall svlm_prefill_small_plan(const SvlmAttendBatch& b, int call_layers, int n_q, int q_heads, const SvlmPrefillLoad* held);
cudaError_t svlm_launch_prefill_small(const SvlmAttendBatch& b, int layer0, int n_layers, const void* Q, const int* q_pos,
                                      int n_q, int q_heads, SvlmPrefillSmall how, void* out, cudaStream_t st);
size_t svlm_prefill_slot_bytes(int n_pages, int head_dim);
constexpr size_t svlm_prefill_counter_bytes = 8192;
cudaError_t svlm_launch_prefill(const SvlmAttendBatch& b, int layer0, int n_layers, int call_layers, const void* Q, const int* q_pos,
                                int n_q, int q_heads, void* out, const SvlmPrefillLoad* held, void* counters, void* slots,
                                cudaStream_t st);
