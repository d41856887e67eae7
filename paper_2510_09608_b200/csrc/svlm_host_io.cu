// Small transfers of the host-buffer entry points as kernels in the cache's stream, instead of copy-engine commands and a
// stream synchronisation: a decode step of one layer moves 10 KB in and 7 KB out, and every hand-over between a copy engine
// and a kernel, and the wake-up from the synchronisation, takes longer than the step.  Reading and writing page-locked host
// memory in place is bound by the bus round trip (about 2 us); the kernels are chained (programmatic dependent launch) to
// the step between them.  svlm_decode_step_host, one layer: 34.9 -> 31.3 us, most of what is left being the start of an idle GPU.
#include <cuda_runtime.h>

#include "svlm_launch.h"
#include "svlm_ptx.cuh"

namespace {

constexpr int IO_THREADS = 256;

// host -> device, 16 bytes per thread; .cv: what the host wrote since the last time must be seen
__global__ void __launch_bounds__(IO_THREADS) host_in_kernel(uint4* __restrict__ dst, const uint4* src, int n16) {
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    const int i = blockIdx.x * IO_THREADS + threadIdx.x;
    if (i < n16) dst[i] = __ldcv(src + i);
}

// device -> host, then the ticket that the host is waiting for (also without anything to copy: everything before this
// kernel in the stream is complete then)
__global__ void __launch_bounds__(IO_THREADS) host_out_kernel(uint4* __restrict__ dst, const uint4* src, int n16, volatile unsigned* done,
                                                             unsigned ticket) {
    svlm_ptx::pdl_wait();
    svlm_ptx::pdl_launch_dependents();
    for (int i = threadIdx.x; i < n16; i += IO_THREADS) dst[i] = svlm_ptx::ld_l2(src + i);
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) *done = ticket;
}

}  // namespace

cudaError_t svlm_launch_host_in(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    const int n16 = (int)((bytes + 15) / 16);
    return svlm_launch_chained(host_in_kernel, dim3((n16 + IO_THREADS - 1) / IO_THREADS), dim3(IO_THREADS), 0, 1, st, static_cast<uint4*>(dst),
                               static_cast<const uint4*>(src), n16);
}

cudaError_t svlm_launch_host_out(void* dst, const void* src, size_t bytes, unsigned* done, unsigned ticket, cudaStream_t st) {
    return svlm_launch_chained(host_out_kernel, dim3(1), dim3(IO_THREADS), 0, 1, st, static_cast<uint4*>(dst), static_cast<const uint4*>(src),
                               (int)((bytes + 15) / 16), done, ticket);
}
