// A stand-in for the CUDA runtime, for tests of the library's host side on a machine without a GPU: device memory is host
// memory, launches are written down instead of run, and calls can be made to fail.  Loaded with global symbols before the
// library, so that the library's references bind here.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::map<const void*, std::string> g_names;
std::string g_log, g_fail;
cudaError_t g_last = cudaSuccess;
size_t g_alloc_limit = ~(size_t)0;
int g_capturing = 0, g_mapped = 0, g_waits = 0;
cudaError_t done(cudaError_t e) { if (e != cudaSuccess) g_last = e; return e; }
cudaError_t launch(const void* f, dim3 grid, dim3 block) {
    const std::string& name = g_names[f];
    if (!g_fail.empty() && name.find(g_fail) != std::string::npos) return done(cudaErrorLaunchOutOfResources);
    g_log += name + " " + std::to_string(grid.x) + "," + std::to_string(grid.y) + "," + std::to_string(grid.z) + " " + std::to_string(block.x) + "\n";
    return cudaSuccess;
}
int encode_nothing() { return 0; }
}  // namespace

extern "C" {
// ---- for the test ----
void fake_fail(const char* kernel) { g_fail = kernel; }          // launches of kernels with this in their name fail
const char* fake_log() { static std::string out; out = g_log; g_log.clear(); return out.c_str(); }   // launches since the last call
void fake_alloc_limit(size_t bytes) { g_alloc_limit = bytes; }   // allocations above this size fail
void fake_capturing(int on) { g_capturing = on; }                // the streams are being captured
void fake_mapped(int on) { g_mapped = on; }                      // host memory is page-locked and mapped
int fake_waits() { const int n = g_waits; g_waits = 0; return n; }   // streams that were made to wait for an event since the last call

// ---- the runtime's calls that the library makes ----
static dim3 g_grid, g_block;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t, void*) { g_grid = grid; g_block = block; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
    *grid = g_grid; *block = g_block; *smem = 0; *static_cast<void**>(stream) = nullptr;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* p; return &p; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) { g_names[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void**, size_t, cudaStream_t) { return launch(f, grid, block); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->gridDim, c->blockDim); }
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = n > g_alloc_limit ? nullptr : std::calloc(1, n);      // (zeros that cost nothing until they are touched)
    return done(*p ? cudaSuccess : cudaErrorMemoryAllocation);
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }                  // the library clears fresh memory only
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { std::memset(a, 0, sizeof *a); a->numRegs = 168; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { ++g_waits; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    if (g_mapped) { a->type = cudaMemoryTypeHost; a->devicePointer = const_cast<void*>(p); }
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** f, unsigned long long, cudaDriverEntryPointQueryResult* r) {
    *f = reinterpret_cast<void*>(encode_nothing);
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}
