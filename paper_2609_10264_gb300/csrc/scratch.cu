// Host-side state kept per device.
//
// Grow-only device scratch held per (purpose, device, stream).
//
// The batched products' digit tiles and the small-batch product's digit
// planes live in one library-owned buffer a stream: every kernel that writes
// it waits for the kernel before, and a call that has sized it serves every
// smaller one, whichever of the two paths that takes.  Keying by stream lets calls on
// different streams overlap without sharing a buffer; calls on one stream
// are ordered, so they may share one.  A buffer that must grow is replaced by
// one of at least twice its size and kept beside it, since kernels in flight
// and captured graphs may still use it; the kept ones come to less than the
// one in use.  Where memory is short those that no capture has been handed
// are given back, after the stream has drained, for a buffer of just the size
// that is needed; a graph may be replayed at any time, so a buffer that one was
// handed is kept for good, and the call is refused if that leaves too little.  A
// buffer cannot grow while the stream is being captured: make one call of the
// largest shape before capturing.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "launch.h"

namespace pv {

namespace {
struct Buf {
    void *ptr = nullptr;
    size_t bytes = 0;
    bool captured = false;    // handed to a call under capture
    std::vector<void *> old;  // outgrown, of no capture
};
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
        size_t bytes = std::max(need, 2 * b.bytes);
        void *p = nullptr;
        e = cudaMalloc(&p, bytes);
        if (e == cudaErrorMemoryAllocation) {
            (void)cudaGetLastError();
            if ((b.ptr && !b.captured) || !b.old.empty()) {
                if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
                for (void *o : b.old) cudaFree(o);
                b.old.clear();
                if (!b.captured) {
                    cudaFree(b.ptr);
                    b.ptr = nullptr;
                    b.bytes = 0;
                }
            }
            e = cudaMalloc(&p, bytes = need);
        }
        if (e != cudaSuccess) return e;
        if (b.ptr && !b.captured) b.old.push_back(b.ptr);
        b.ptr = p;
        b.bytes = bytes;
        b.captured = false;
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
