// The CUDA runtime functions and kernel launchers that kvs_api.cpp calls, as stand-ins that
// do nothing but write down the launches: the planner's choices can then be tested without
// a GPU.  An event pair that encloses a launch of kernel k is fake_set_ms(k)'s time long.
#include <cstdlib>
#include <vector>

#include <cuda.h>
#include <cuda_runtime.h>

#include "kvs_internal.h"

namespace {
enum Kernel { LDG, TMA, LINK, LINK_STAGED, LINK_PREFETCH, LINK_SIGNAL, FP8_RETRIEVE, FP8_RETRIEVE_STAGED, FP8_STORE, OTHER };
struct Launch {
    int kernel, grid, carried, early;
};
std::vector<Launch> g_seen;
float g_ms[OTHER + 1];
int g_last = OTHER;

cudaError_t launched(int kernel, const kvs::Job& j, int grid) {
    g_last = kernel;
    g_seen.push_back({kernel, grid, j.tables != nullptr, (int)j.early});
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset() {
    g_seen.clear();
    for (float& m : g_ms) m = 1.0f;
}
void fake_set_ms(int kernel, float ms) { g_ms[kernel] = ms; }
int fake_count() { return (int)g_seen.size(); }
void fake_launch(int k, int* out) {
    const Launch& l = g_seen[k];
    const int v[] = {l.kernel, l.grid, l.carried, l.early};
    for (size_t i = 0; i < sizeof v / sizeof *v; ++i) out[i] = v[i];
}

cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1 << 30;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)1, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = g_ms[g_last], cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *f = nullptr;
    *q = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)1, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) { return *c = cudaStreamCaptureStatusNone, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
}

namespace kvs {
int kernels_of(const Job&, int) { return 1; }
int link_ctas_per_sm() { return 3; }
void noalloc_forget_devices() {}
cudaError_t launch_ldg(const Job& j, int, int grid, cudaStream_t) { return launched(LDG, j, grid); }
cudaError_t launch_tma(const Job& j, int grid, cudaStream_t) { return launched(TMA, j, grid); }
cudaError_t launch_link(const Job& j, int, int grid, cudaStream_t) { return launched(LINK, j, grid); }
cudaError_t launch_link_staged(const Job& j, int grid, cudaStream_t) { return launched(LINK_STAGED, j, grid); }
cudaError_t launch_link_prefetch(const Job& j, int grid, cudaStream_t) { return launched(LINK_PREFETCH, j, grid); }
cudaError_t launch_link_signal(const Job& j, const Signal&, int grid, cudaStream_t) { return launched(LINK_SIGNAL, j, grid); }
cudaError_t launch_fp8_retrieve(const Fp8Job& f, int grid, cudaStream_t) { return launched(FP8_RETRIEVE, f.job, grid); }
cudaError_t launch_fp8_retrieve_staged(const Fp8Job& f, int grid, cudaStream_t) { return launched(FP8_RETRIEVE_STAGED, f.job, grid); }
cudaError_t launch_fp8_store(const Fp8Job& f, int grid, cudaStream_t, uint32_t, bool) { return launched(FP8_STORE, f.job, grid); }
cudaError_t launch_stall(int32_t*, uint64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_flat_copy(void*, const void*, uint64_t, int, cudaStream_t) { return g_last = OTHER, cudaSuccess; }
}  // namespace kvs
