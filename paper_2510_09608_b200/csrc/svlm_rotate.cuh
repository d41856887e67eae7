// Rotating eight pairs of a key, shared by the kernels that write keys (svlm_kv.cu) and by the metadata kernels of small
// caches, which do it themselves (svlm_meta.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include "svlm_dev.h"
#include "svlm_rope.cuh"

namespace {

struct __align__(16) Bf16x8 { __nv_bfloat162 v[4]; };
__device__ __forceinline__ Bf16x8 bf16x8(const uint4& x) { return reinterpret_cast<const Bf16x8&>(x); }

// Rotate 8 consecutive pairs (lo[j], hi[j]) by (cs[j], sn[j]) in fp32, round to bf16.
__device__ __forceinline__ void rotate8(Bf16x8& lo, Bf16x8& hi, const float* cs, const float* sn) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 a = __bfloat1622float2(lo.v[j]);
        const float2 b = __bfloat1622float2(hi.v[j]);
        float2 ra, rb;
        ra.x = a.x * cs[2 * j] - b.x * sn[2 * j];
        rb.x = b.x * cs[2 * j] + a.x * sn[2 * j];
        ra.y = a.y * cs[2 * j + 1] - b.y * sn[2 * j + 1];
        rb.y = b.y * cs[2 * j + 1] + a.y * sn[2 * j + 1];
        lo.v[j] = __float22bfloat162_rn(ra);
        hi.v[j] = __float22bfloat162_rn(rb);
    }
}

// Factors of pairs 8 g .. 8 g + 7 of a token at positions c.
__device__ __forceinline__ void first_rotation(const SvlmCacheDev& cd, int g, const int (&c)[3], float (&cs)[8], float (&sn)[8]) {
    const int half = cd.head_dim / 2;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int pair = g * 8 + j;
        const int axis = cd.rope_mode == 0 ? 0 : (pair < cd.sec_t ? 0 : (pair < cd.sec_th ? 1 : 2));
        const float2 f = svlm_rope_cs_batched(reinterpret_cast<const float2*>(cd.rope_tab), half, pair, axis == 0 ? c[0] : (axis == 1 ? c[1] : c[2]));
        cs[j] = f.x;
        sn[j] = f.y;
    }
    const int lim = 1 << 16;
    if (c[0] <= -lim || c[0] >= lim || c[1] <= -lim || c[1] >= lim || c[2] <= -lim || c[2] >= lim) {   // native positions of a long stream
#pragma unroll 1
        for (int j = 0; j < 8; ++j) {
            const int pair = g * 8 + j;
            const int axis = cd.rope_mode == 0 ? 0 : (pair < cd.sec_t ? 0 : (pair < cd.sec_th ? 1 : 2));
            const float2 f = svlm_rope_cs(reinterpret_cast<const float2*>(cd.rope_tab), half, pair, axis == 0 ? c[0] : (axis == 1 ? c[1] : c[2]), cd.theta[pair]);
#pragma unroll
            for (int q = 0; q < 8; ++q) if (q == j) { cs[q] = f.x; sn[q] = f.y; }
        }
    }
}

}  // namespace
