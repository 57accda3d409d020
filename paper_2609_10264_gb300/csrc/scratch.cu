// Host-side state kept per device.
//
// Grow-only device scratch held per (purpose, device, stream).
//
// The batched products' digit tiles and the small-batch product's digit
// planes live in one library-owned buffer a stream: every kernel that writes
// it waits for the kernel before, and a call that has sized it serves every
// smaller one, whichever of the two paths that takes.  Keying by stream lets calls on
// different streams overlap without sharing a buffer; calls on one stream
// are ordered, so they may share one.  A buffer that must grow is given back
// once the stream has drained; one that a captured call was handed is kept
// for good instead, since its graph may be replayed at any time, and then the
// new one has at least twice its size, so that those kept come to less than the
// one in use.  Otherwise growth is rounded up by kGrowSlack at most.  Where that
// is not to be had the call gets just what it needs, or is refused.  A buffer
// cannot grow while the stream is being captured: make one call of the
// largest shape before capturing.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "launch.h"

namespace pv {

namespace {
struct Buf {
    void *ptr = nullptr;
    size_t bytes = 0;
    bool captured = false;  // handed to a call under capture
};
constexpr size_t kGrowSlack = 32u << 20;
std::mutex g_bufs_mu;
std::map<std::tuple<int, int, cudaStream_t>, Buf> g_bufs;
}  // namespace

bool stream_scratch_ready(int purpose, size_t need, cudaStream_t s) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    {
        std::lock_guard<std::mutex> lock(g_bufs_mu);
        const auto it = g_bufs.find(std::make_tuple(purpose, dev, s));
        if (it != g_bufs.end() && it->second.bytes >= need) return true;
    }
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone;
}

cudaError_t stream_scratch(int purpose, size_t need, cudaStream_t s, void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_bufs_mu);
    Buf &b = g_bufs[std::make_tuple(purpose, dev, s)];
    if (b.bytes < need) {
        size_t bytes = std::max(need, b.captured ? 2 * b.bytes : std::min(2 * b.bytes, b.bytes + kGrowSlack));
        void *p = nullptr;
        if (b.ptr && !b.captured) {
            if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
            cudaFree(b.ptr);
            b = Buf{};
        }
        e = cudaMalloc(&p, bytes);
        if (e == cudaErrorMemoryAllocation && bytes > need) {
            (void)cudaGetLastError();
            e = cudaMalloc(&p, bytes = need);
        }
        if (e != cudaSuccess) return e;
        b = Buf{p, bytes, false};
    }
    if (!b.captured) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {  // the legacy stream, while another is captured
            (void)cudaGetLastError();
            capture = cudaStreamCaptureStatusActive;
        }
        b.captured = capture != cudaStreamCaptureStatusNone;
    }
    *out = b.ptr;
    return cudaSuccess;
}

cudaError_t func_attr(const void *fn, cudaFuncAttribute attr, int value) {
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, int>, std::pair<int, cudaError_t>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    auto key = std::make_tuple(fn, (int)attr, dev);
    auto it = done.find(key);
    if (it != done.end() && it->second.first == value) return it->second.second;
    e = cudaFuncSetAttribute(fn, attr, value);
    done[key] = std::make_pair(value, e);
    return e;
}

}  // namespace pv
