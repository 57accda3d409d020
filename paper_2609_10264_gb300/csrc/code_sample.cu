// Device sampling of the public RAA codes (App. B): the permutations pi1, pi2
// and the scalings v1, v2 of a code, and the tables the kernels read.  The
// sampler's specification is that of sample_code_host (api.cu), draw for draw.
//
//  * k_code_draws   one CTA per array: the field draws of v1 and v2, and the
//                   Fisher-Yates indices j_i <= i of pi1 and pi2.
//  * k_perm_link, k_perm_next, k_code_tables
//                   the permutation those swaps give, without doing them in
//                   order, and the derived tables.
//
// A swap (i, j_i), i = N-1 .. 1, settles position i: a[i] becomes the value at
// j_i, and j_i receives the value that was at i.  So the value at position p
// before step i is the one that the latest step i' > i with j_i' = p (the
// smallest such i') moved there, which is the value at i' before step i', and p
// itself where there is no such step.  With next(p) the smallest i' > p that
// drew p, the value V(p) at p before step p is found by following next to its
// end (a chain of O(log N) steps), and a[i] = V(i') for the smallest i' > i that
// drew j_i, else j_i.  The steps that drew a position are a linked list (one on
// average).
//
// Latency-bound, a few kernels of 10 to 100 us for any N; one host thread took
// 1.3 ms per code at N = 32768, and its tables and their copies about as much.
#include "common.cuh"
#include "launch.h"

namespace pv {
namespace {

constexpr int kDrawThreads = 1024;
constexpr uint32_t kNone = 0xffffffffu;
constexpr uint32_t kRound = kDrawThreads * 16;  // keystream words per round: a block per thread

struct DrawArgs {
    pvmvmd_key key;
    CodeDraws code[2];
};

// The keystream words [16 * kDrawThreads * round, ...) of stream (tag, 0).
__device__ __forceinline__ void draw_words(const pvmvmd_key &key, uint32_t tag, uint32_t round, uint32_t out[16]) {
    chacha20_block_dev(key, round * kDrawThreads + threadIdx.x, tag, 0u, 0u, out);
}

__device__ void draw_field(const pvmvmd_key &key, uint32_t tag, uint32_t N, uint32_t *__restrict__ out,
                           uint32_t *s_wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t have = 0;
    for (uint32_t round = 0; have < N; ++round) {
        uint32_t w[16], c = 0;
        draw_words(key, tag, round, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            w[i] >>= 1;
            c += w[i] != 0u && w[i] < kQ;
        }
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        const uint32_t wv = s_wsum[lane];  // 32 warps
        uint32_t pos = have + __reduce_add_sync(kFull, lane < warp ? wv : 0u) + incl - c;
        have += __reduce_add_sync(kFull, wv);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (w[i] != 0u && w[i] < kQ) {
                if (pos < N) out[pos] = w[i];
                ++pos;
            }
    }
}

__device__ __forceinline__ bool index_draw(uint32_t word, uint32_t i, uint32_t &v) {
    v = word >> __clz(i);  // the top bitlen(i) bits, i >= 1
    return v <= i;
}

// j[i] for i = N-1 .. 1: a word is accepted or not against the i its
// predecessors leave, so the flags of a batch are iterated to their fixed
// point: a word's flag rests on the words before it alone, so the fixed point
// is unique, and one more word is settled by every turn at least; since i
// moves by less than 1024 in a batch while draws range over more than 2048
// values, two or three turns settle it.  The last 2048 indices are drawn by
// one warp, 32 words at a time.
__device__ void draw_swaps(const pvmvmd_key &key, uint32_t tag, uint32_t N, uint32_t *__restrict__ j, uint32_t *s_words,
                           uint32_t *s_wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t left = N - 1;  // the next index to draw (N >= 1); 0: done
    for (uint32_t round = 0; left > 0; ++round) {
        uint32_t blk[16];
        draw_words(key, tag, round, blk);
        __syncthreads();  // the words of the round before are no longer read
#pragma unroll
        for (int i = 0; i < 16; ++i) s_words[tid * 16 + i] = blk[i];
        __syncthreads();
        uint32_t at = 0;
        for (; at < kRound && left >= 2048; at += kDrawThreads) {
            const uint32_t word = s_words[at + tid];
            uint32_t v, before = 0, total = 0;
            bool flag = index_draw(word, left, v);
            for (;;) {
                const uint32_t mask = __ballot_sync(kFull, flag);
                if (lane == 0) s_wsum[warp] = __popc(mask);
                __syncthreads();
                const uint32_t wv = s_wsum[lane];
                before = __reduce_add_sync(kFull, lane < warp ? wv : 0u) + __popc(mask & lanemask_lt());
                total = __reduce_add_sync(kFull, wv);
                const bool now = index_draw(word, left - before, v);
                const bool changed = now != flag;
                flag = now;
                if (!__syncthreads_or(changed)) break;
            }
            if (flag) j[left - before] = v;
            left -= total;
        }
        if (left >= 2048) continue;
        if (warp == 0) {
            for (; at < kRound && left > 0; at += 32) {
                const uint32_t word = s_words[at + lane];
                uint32_t v, before = 0, mask = 0;
                bool flag = index_draw(word, left, v);
                for (;;) {
                    mask = __ballot_sync(kFull, flag);
                    before = __popc(mask & lanemask_lt());
                    const bool now = before < left && index_draw(word, left - before, v);
                    const bool changed = now != flag;
                    flag = now;
                    if (!__any_sync(kFull, changed)) break;
                }
                if (flag) j[left - before] = v;
                left -= __popc(mask);
            }
            if (lane == 0) s_wsum[0] = left;
        }
        __syncthreads();
        left = s_wsum[0];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kDrawThreads) k_code_draws(const DrawArgs args) {
    extern __shared__ uint32_t s_words[];
    __shared__ uint32_t s_wsum[32];
    const CodeDraws &c = args.code[blockIdx.y];
    // tags: pi1, pi2, v1, v2
    if (blockIdx.x < 2) draw_swaps(args.key, c.tag0 + blockIdx.x, c.N, c.perm[blockIdx.x].j, s_words, s_wsum);
    else draw_field(args.key, c.tag0 + blockIdx.x, c.N, blockIdx.x == 2 ? c.v1 : c.v2, s_wsum);
}

// list of the steps i >= 1 that drew a position
__global__ void __launch_bounds__(256) k_perm_link(const DrawArgs args) {
    const CodeDraws &c = args.code[blockIdx.z];
    const PermScratch &p = c.perm[blockIdx.y];
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i >= 1 && i < c.N) p.link[i] = atomicExch(p.head + p.j[i], i);
    if (i == 0) p.j[0] = 0;  // the last index is never drawn
}

// next[i]: the smallest step after i that drew i; succ[i]: that drew j_i
__global__ void __launch_bounds__(256) k_perm_next(const DrawArgs args) {
    const CodeDraws &c = args.code[blockIdx.z];
    const PermScratch &p = c.perm[blockIdx.y];
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i >= c.N) return;
    auto after = [&](uint32_t pos) {
        uint32_t best = kNone;
        for (uint32_t e = p.head[pos]; e != kNone; e = p.link[e])
            if (e > i && e < best) best = e;
        return best;
    };
    p.next[i] = after(i);
    p.succ[i] = after(p.j[i]);
}

__global__ void __launch_bounds__(256) k_code_tables(const DrawArgs args) {
    const CodeDraws &c = args.code[blockIdx.z];
    const PermScratch &p = c.perm[blockIdx.y];
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i >= c.N) return;
    uint32_t a = p.j[i];
    uint32_t e = p.succ[i];
    while (e != kNone) {
        a = e;
        e = p.next[e];
    }
    const bool first = blockIdx.y == 0;
    const uint32_t v = first ? c.v1[i] : c.v2[i], vm = (uint32_t)(((uint64_t)v << 32) % kQ);
    if (first) {
        c.pi1[i] = a;
        c.pi1inv[a] = i;
        c.v1m[i] = vm;
        c.v1pm[a] = vm;
    } else {
        c.pi2[i] = a;
        c.pi2inv[a] = i;
        c.v2m[i] = vm;
        c.v2p[a] = v;
    }
}

}  // namespace

size_t code_draw_scratch_words(uint32_t N) { return 2 * 5 * (size_t)N; }

cudaError_t launch_code_draws(const pvmvmd_key &key, CodeDraws *codes, int count, uint32_t *const *scratch,
                              cudaStream_t s) {
    DrawArgs args{};
    args.key = key;
    uint32_t most = 0;
    for (int k = 0; k < count; ++k) {
        CodeDraws &c = codes[k];
        if (c.N == 0) return cudaErrorInvalidValue;
        // the two heads first: one fill clears both
        const cudaError_t e = cudaMemsetAsync(scratch[k], 0xff, 2 * (size_t)c.N * sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        for (int p = 0; p < 2; ++p) {
            uint32_t *base = scratch[k] + (2 + 4 * (size_t)p) * c.N;
            c.perm[p] = PermScratch{base, scratch[k] + (size_t)p * c.N, base + c.N, base + 2 * (size_t)c.N,
                                    base + 3 * (size_t)c.N};
        }
        args.code[k] = c;
        most = c.N > most ? c.N : most;
    }
    const cudaError_t attr = func_attr((const void *)k_code_draws, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(kRound * sizeof(uint32_t)));
    if (attr != cudaSuccess) return attr;
    k_code_draws<<<dim3(4, count), kDrawThreads, kRound * sizeof(uint32_t), s>>>(args); note_launch();
    const dim3 grid((most + 255) / 256, 2, count);
    k_perm_link<<<grid, 256, 0, s>>>(args); note_launch();
    k_perm_next<<<grid, 256, 0, s>>>(args); note_launch();
    k_code_tables<<<grid, 256, 0, s>>>(args); note_launch();
    return cudaGetLastError();
}

}  // namespace pv
