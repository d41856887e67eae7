// Inline-PTX wrappers shared by the sm_100a kernels: mbarriers with bounded waits, TMA tile loads,
// proxy fences, programmatic-dependent-launch controls.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace svlm_ptx {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(void* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(void* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(void* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(void* bar, unsigned parity) {
    unsigned ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: false when `limit` polls ran out (a limit of 0 gives up at once, whatever the barrier's
// state) or another thread of the CTA already gave up.
__device__ __forceinline__ bool mbar_wait(void* bar, unsigned parity, volatile int* abort_flag, unsigned limit) {
    for (unsigned it = 0; it < limit; ++it) {
        if (mbar_test(bar, parity)) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            __nanosleep(64);
        }
    }
    *abort_flag = 1;
    return false;
}
// `n` polls at most; a loop of few instructions, since what a wait costs is less the barrier than the fetching of its code.
__device__ __forceinline__ bool mbar_poll(unsigned bar, unsigned parity, unsigned n) {
    unsigned ok;
    asm volatile("{\n.reg .pred p, q;\n.reg .u32 n;\nmov.u32 n, %3;\nsetp.ne.u32 p, 0, 0;\n"
                 "setp.eq.u32 q, n, 0;\n@q bra DONE;\n"
                 "LOOP:\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n@p bra DONE;\n"
                 "sub.u32 n, n, 1;\nsetp.ne.u32 q, n, 0;\n@q bra LOOP;\n"
                 "DONE:\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(n) : "memory");
    return ok != 0;
}
// mbar_wait for a whole warp (all lanes poll: no branch by lane, nothing to hand around afterwards).
__device__ __forceinline__ bool mbar_wait_short(void* bar, unsigned parity, volatile int* abort_flag, unsigned limit) {
    const unsigned b = smem_u32(bar);
#pragma unroll 1
    while (!mbar_poll(b, parity, min(limit, 64u))) {
        limit -= min(limit, 64u);
        if (limit == 0 || *abort_flag) {
            *abort_flag = 1;
            return false;
        }
        __nanosleep(64);
    }
    return true;
}
// 2D tiled TMA load into this CTA's shared memory; completion is counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, int x, int y, void* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
// For loads of data that a pass over the layers reads once, a layer's weights: the first to make room in L2.  They are more than what
// else a layer touches, and what comes again with the next layer (code, tables, activations) stays.
__device__ __forceinline__ unsigned long long l2_read_once() {
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
// The same tile only brought into L2 (no shared memory, no barrier): for data whose stage is not free yet.
__device__ __forceinline__ void tma_prefetch_2d(const void* tmap, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tmap), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Fragments of mma.sync from shared memory, and the instruction (bf16 in, fp32 accumulation).
__device__ __forceinline__ void ldmatrix_x4(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3, const void* p) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(s));
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3,
                                                  const void* p) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(s));
}
__device__ __forceinline__ void mma_bf16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Loads of what an earlier kernel of the stream writes.  With programmatic dependent launch that kernel may still be running
// when this one starts, so such data must not take the read-only path (ld.global.nc, which __ldg and const __restrict__
// parameters allow: it is for data that nobody writes while the kernel runs, and the compiler may move such a load above
// the wait).  These are volatile and stay behind pdl_wait().  ld_l2 reads past L1.
#define SVLM_LOAD(name, T, instr, reg)                                       \
    __device__ __forceinline__ T name(const T* p) {                         \
        T v;                                                                \
        asm volatile(instr " %0, [%1];" : reg(v) : "l"(p) : "memory");      \
        return v;                                                           \
    }
#define SVLM_LOAD2(name, T, instr, reg)                                                             \
    __device__ __forceinline__ T name(const T* p) {                                                 \
        T v;                                                                                        \
        asm volatile(instr " {%0, %1}, [%2];" : reg(v.x), reg(v.y) : "l"(p) : "memory");            \
        return v;                                                                                   \
    }
#define SVLM_LOAD4(name, T, instr, reg)                                                                                             \
    __device__ __forceinline__ T name(const T* p) {                                                                                 \
        T v;                                                                                                                        \
        asm volatile(instr " {%0, %1, %2, %3}, [%4];" : reg(v.x), reg(v.y), reg(v.z), reg(v.w) : "l"(p) : "memory");                \
        return v;                                                                                                                   \
    }
SVLM_LOAD(ld_in, uint16_t, "ld.global.u16", "=h")
SVLM_LOAD(ld_in, int, "ld.global.s32", "=r")
SVLM_LOAD(ld_in, unsigned, "ld.global.u32", "=r")
SVLM_LOAD2(ld_in, longlong2, "ld.global.v2.s64", "=l")
SVLM_LOAD4(ld_in, uint4, "ld.global.v4.u32", "=r")
SVLM_LOAD(ld_l2, int, "ld.global.cg.s32", "=r")
SVLM_LOAD(ld_l2, unsigned, "ld.global.cg.u32", "=r")
SVLM_LOAD(ld_l2, long long, "ld.global.cg.s64", "=l")
SVLM_LOAD2(ld_l2, longlong2, "ld.global.cg.v2.s64", "=l")
SVLM_LOAD2(ld_l2, float2, "ld.global.cg.v2.f32", "=f")
SVLM_LOAD4(ld_l2, float4, "ld.global.cg.v4.f32", "=f")
SVLM_LOAD4(ld_l2, int4, "ld.global.cg.v4.s32", "=r")
SVLM_LOAD4(ld_l2, uint4, "ld.global.cg.v4.u32", "=r")
__device__ __forceinline__ unsigned char ld_in(const unsigned char* p) {
    unsigned v;
    asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return (unsigned char)v;
}
#undef SVLM_LOAD
#undef SVLM_LOAD2
#undef SVLM_LOAD4

// Programmatic dependent launch: let the next kernel in the stream start; wait for the previous one.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace svlm_ptx
