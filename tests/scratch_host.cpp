// csrc/scratch.cu on the host, against a pretended CUDA runtime: a device of a
// given size whose streams may be said to be capturing.  Driven by
// test_scratch_host.py.
#include <cstdlib>
#include <map>

#include <cuda_runtime.h>

namespace {
std::map<void *, size_t> g_live;
size_t g_used = 0, g_size = 0;
bool g_capturing = false;
int g_syncs = 0;
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *dev) {
    *dev = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
    if (g_capturing) return cudaErrorStreamCaptureUnsupported;
    if (g_used + n > g_size) return cudaErrorMemoryAllocation;
    *p = std::malloc(1);  // an address of its own
    g_live[*p] = n;
    g_used += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    const auto it = g_live.find(p);
    if (it == g_live.end()) return cudaErrorInvalidValue;
    g_used -= it->second;
    g_live.erase(it);  // the address is not given out again
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    if (g_capturing) return cudaErrorStreamCaptureUnsupported;
    ++g_syncs;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
}

#include "scratch.cu"

extern "C" {
void host_reset(size_t size) {
    for (const auto &b : g_live) std::free(b.first);
    g_live.clear();
    pv::g_bufs.clear();
    g_used = 0;
    g_size = size;
    g_capturing = false;
    g_syncs = 0;
}
void host_capturing(int on) { g_capturing = on != 0; }
size_t host_used(void) { return g_used; }
int host_syncs(void) { return g_syncs; }
int host_live(void *p) { return g_live.count(p) != 0; }
int host_scratch(size_t need, void **out) { return pv::stream_scratch(pv::kScratchDigits, need, nullptr, out); }
}
