// The host side of a decode (csrc/api.cu) against a pretended CUDA runtime that
// writes down what is enqueued where and fails one step on request.
//   decode_host CALL...     CALL: kind[:step], kind one of side, caller, inplace,
//                           captured; step the number of the enqueueing step
//                           that fails
// prints one line per step and one per call's status.  Driven by
// test_decode_host.py.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include <cuda_runtime.h>

// named by device code that is compiled for the host here and never run
template <typename T> T __ldg(const T *p) { return *p; }
template <typename T> T __ldcg(const T *p) { return *p; }
static inline unsigned __funnelshift_l(unsigned, unsigned, unsigned) { return 0; }
static inline unsigned __funnelshift_r(unsigned, unsigned, unsigned) { return 0; }
static inline unsigned atomicOr(unsigned *, unsigned) { return 0; }
static inline cudaError_t cudaGetSymbolAddress(void **p, unsigned &word) {
    *p = &word;
    return cudaSuccess;
}

#include "api.cu"

namespace {
int g_step = 0, g_fail = -1;
bool g_capturing = false, g_large = false;
const char *name(const void *s) { return s == (const void *)1 ? "caller" : s == (const void *)2 ? "side" : "other"; }
bool step(const char *what, const void *s) {
    const bool bad = g_step++ == g_fail;
    std::printf("%s %s%s\n", what, name(s), bad ? " failed" : "");
    return !bad;
}
cudaError_t enqueue(const char *what, const void *s) { return step(what, s) ? cudaSuccess : cudaErrorUnknown; }
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    return enqueue(e == (cudaEvent_t)3 ? "record fork" : "record join", s);
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    return enqueue(e == (cudaEvent_t)3 ? "wait fork" : "wait join", s);
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::printf("synchronize %s\n", name(s));
    return cudaSuccess;
}
}

namespace pv {
bool syndrome_tiles_eligible(uint32_t) { return true; }
bool decode_wins(int, int, uint32_t, uint32_t, uint32_t) { return g_large; }
cudaError_t launch_decode(const DecodeCall &, cudaStream_t s) { return enqueue("decode", s); }
cudaError_t launch_syndrome_tiles(const pvmvmd_key &, uint32_t, uint64_t, uint32_t, uint32_t, uint32_t, const uint32_t *,
                                  const uint32_t *, const uint32_t *, const uint32_t *, uint32_t, uint32_t, uint32_t *,
                                  uint32_t *, unsigned long long *, uint32_t *, const uint32_t *, uint32_t *,
                                  cudaStream_t s, bool, const uint32_t *, int, uint32_t *) {
    return enqueue("challenges", s);
}
cudaError_t launch_check(const uint32_t *, int, const uint32_t *, int, const uint32_t *, const uint32_t *, uint32_t, int,
                         int32_t *, cudaStream_t s) {
    return enqueue("check", s);
}
cudaError_t launch_decrypt(const uint32_t *, int, const uint32_t *, uint32_t, uint32_t, const uint32_t *, int,
                           uint32_t *, cudaStream_t s, const uint32_t *) {
    return enqueue("decrypt", s);
}
}  // namespace pv

int main(int argc, char **argv) {
    pvmvmd_ctx ctx;
    ctx.m = ctx.K = 4;
    ctx.side = (cudaStream_t)2;
    ctx.fork = (cudaEvent_t)3;
    ctx.join = (cudaEvent_t)4;
    uint32_t st[8], x[4], y[4], out[4];
    int32_t acc[1];
    const pvmvmd_key key{};
    for (int i = 1; i < argc; ++i) {
        const char *colon = std::strchr(argv[i], ':');
        g_fail = colon ? std::atoi(colon + 1) : -1;
        g_step = 0;
        g_large = std::strncmp(argv[i], "caller", 6) == 0;
        g_capturing = std::strncmp(argv[i], "captured", 8) == 0;
        uint32_t *Y = std::strncmp(argv[i], "inplace", 7) == 0 ? y : out;
        std::printf("status %d\n", pvmvmd_decode_verify(&ctx, st, x, y, 1, &key, Y, acc, (void *)1));
    }
    return 0;
}
