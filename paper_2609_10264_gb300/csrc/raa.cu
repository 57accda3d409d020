// RAA code kernels (App. B of the paper) and the sparse sampler.
//
//  * k_sample_sparse      draws e <- E_t^N (Sec. 3 notation) on the device.
//  * k_syndrome_scan      first half of the syndrome x' = G e for a sparse e:
//                         step function A e, permutation, and the suffix-sum
//                         accumulator as a single-pass decoupled look-back scan.
//  * k_syndrome_gather    second half: inverse permutation gather and the
//                         block sums of R, fused with x_hat = x + x'.
//  * k_syndrome_fused     the whole syndrome, a vector per CTA with its code in
//                         shared memory.
//  * k_syndrome_sliced    the same for longer codes and many vectors, slice by
//                         slice (k_slice_tables orders the positions).
//  * k_syndrome_tiles     the syndrome's first half for a few vectors, or a few
//                         shared challenges: every CTA samples e itself and
//                         takes one tile of 2048 positions.
//  * k_encode_scan        one accumulate stage of the encoding G^T w over many
//                         lanes (preprocessing of P^T and Q, Sec. 6.3).
//  * k_lane_*             the syndrome for a batch of vectors held as the lanes
//                         of an N x B array (sample, step function, scan, gather).
#include <map>
#include <mutex>
#include "common.cuh"
#include "launch.h"
#include "syndrome.cuh"

namespace pv {
namespace {

// -----------------------------------------------------------------------------
// Sparse sampler: one warp per vector.  Specification (shared with the oracle,
// written independently there): the support is the first t distinct values of
// the sequence below(N) read from the ChaCha20 stream with nonce
// (tag, 2 idx); below(k) keeps the top bitlen(k-1) bits of a 32-bit word and
// rejects values >= k.  Values are the first t words of stream (tag, 2 idx + 1)
// whose top 31 bits lie in [1, q); the k-th one goes to the k-th smallest
// support index.
// -----------------------------------------------------------------------------
// Warp: mark the support of e <- E_t^N in `bitmap` (N bits, cleared by the
// caller) from stream (tag, sidx), using `words` (512 words) as keystream buffer.
__device__ void warp_sample_support(const pvmvmd_key &key, uint32_t tag, uint64_t sidx, uint32_t N,
                                    uint32_t t, uint32_t *bitmap, uint32_t *words, int lane) {
    uint32_t have = 0;
    if (N <= 1) {  // below(1) = 0 reads no word
        if (t >= 1 && lane == 0) bitmap[0] = 1u;
        __syncwarp();
        return;
    }
    const int shift = 32 - bitlen32(N - 1);
    for (uint64_t wpos = 0; have < t; wpos += 512) {
        uint32_t blk[16];
        chacha20_block_dev(key, (uint32_t)(wpos / 16 + lane), tag, (uint32_t)sidx,
                           (uint32_t)(sidx >> 32), blk);
#pragma unroll
        for (int i = 0; i < 16; ++i) words[lane * 16 + i] = blk[i];
        __syncwarp();
        for (int batch = 0; batch < 16 && have < t; ++batch) {
            const uint32_t v = words[batch * 32 + lane] >> shift;
            const bool valid = v < N;
            const bool inset = valid && ((bitmap[v >> 5] >> (v & 31)) & 1u);
            const uint32_t vmask = __ballot_sync(kFull, valid);
            const uint32_t same = __match_any_sync(kFull, valid ? v : 0xffffffffu);
            const bool dup = (same & vmask & lanemask_lt()) != 0u;
            const bool cand = valid && !inset && !dup;
            const uint32_t cmask = __ballot_sync(kFull, cand);
            const uint32_t need = t - have;
            __syncwarp();  // every lane has read the bitmap before it changes
            if (cand && (uint32_t)__popc(cmask & lanemask_lt()) < need)
                atomicOr(&bitmap[v >> 5], 1u << (v & 31));
            have += min((uint32_t)__popc(cmask), need);
            __syncwarp();
        }
        __syncwarp();  // words are read before the next refill
    }
}

// Warp: as warp_sample_support, and also writes the accepted indices, in the
// order they were accepted, to list[0..t).
__device__ void warp_sample_support_list(const pvmvmd_key &key, uint32_t tag, uint64_t sidx,
                                         uint32_t N, uint32_t t, uint32_t *bitmap, uint32_t *words,
                                         uint32_t *list, int lane) {
    uint32_t have = 0;
    if (N <= 1) {
        if (t >= 1 && lane == 0) list[0] = 0u;
        __syncwarp();
        return;
    }
    const int shift = 32 - bitlen32(N - 1);
    for (uint64_t wpos = 0; have < t; wpos += 512) {
        uint32_t blk[16];
        chacha20_block_dev(key, (uint32_t)(wpos / 16 + lane), tag, (uint32_t)sidx,
                           (uint32_t)(sidx >> 32), blk);
#pragma unroll
        for (int i = 0; i < 16; ++i) words[lane * 16 + i] = blk[i];
        __syncwarp();
        for (int batch = 0; batch < 16 && have < t; ++batch) {
            const uint32_t v = words[batch * 32 + lane] >> shift;
            const bool valid = v < N;
            const bool inset = valid && ((bitmap[v >> 5] >> (v & 31)) & 1u);
            const uint32_t vmask = __ballot_sync(kFull, valid);
            const uint32_t same = __match_any_sync(kFull, valid ? v : 0xffffffffu);
            const bool dup = (same & vmask & lanemask_lt()) != 0u;
            const bool cand = valid && !inset && !dup;
            const uint32_t cmask = __ballot_sync(kFull, cand);
            const uint32_t need = t - have;
            const uint32_t rk = __popc(cmask & lanemask_lt());
            __syncwarp();
            if (cand && rk < need) {
                atomicOr(&bitmap[v >> 5], 1u << (v & 31));
                list[have + rk] = v;
            }
            have += min((uint32_t)__popc(cmask), need);
            __syncwarp();
        }
        __syncwarp();
    }
}

// Warp: the set bits of `bitmap` (nbw words) in ascending order -> dst.
__device__ void warp_bitmap_to_support(const uint32_t *bitmap, uint32_t nbw, uint32_t *dst, int lane) {
    uint32_t written = 0;
    for (uint32_t base = 0; base < nbw; base += 32) {
        uint32_t w = (base + lane < nbw) ? bitmap[base + lane] : 0u;
        const uint32_t c = __popc(w);
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t pos = written + incl - c;
        while (w) {
            const int b = __ffs(w) - 1;
            dst[pos++] = (base + lane) * 32 + b;
            w &= w - 1;
        }
        written += __shfl_sync(kFull, incl, 31);
    }
}

// One warp per vector (before k_syndrome_scan).
__global__ void __launch_bounds__(32) k_sample_sparse(pvmvmd_key key, uint32_t tag, uint64_t idx0,
                                                     uint32_t N, uint32_t t,
                                                     uint32_t *__restrict__ out,
                                                     unsigned long long *__restrict__ clear,
                                                     size_t clear_words) {
    extern __shared__ uint32_t sm[];
    const uint32_t nbw = (N + 31) / 32;
    uint32_t *bitmap = sm;
    uint32_t *words = sm + nbw;  // 512 keystream words = 32 blocks
    const int lane = threadIdx.x;

    for (size_t i = (size_t)blockIdx.x * 32 + lane; i < clear_words; i += (size_t)gridDim.x * 32)
        clear[i] = 0ull;

    const uint64_t idx = idx0 + blockIdx.x;
    uint32_t *supp = out + (size_t)blockIdx.x * 2 * t;
    for (uint32_t w = lane; w < nbw; w += 32) bitmap[w] = 0u;
    __syncwarp();
    warp_sample_support(key, tag, 2 * idx, N, t, bitmap, words, lane);
    warp_bitmap_to_support(bitmap, nbw, supp, lane);
    warp_sample_values(key, tag, 2 * idx + 1, t, words, supp + t, lane);
}

// -----------------------------------------------------------------------------
// Syndrome scan.  For sparse e with ascending support s_0 < ... < s_{t-1}:
//   (A e)_k = sum_{s_j >= k} e_j   (A_{i,j} = 1 iff i <= j: suffix sums)
//   c_i     = v2[pi2^-1(i)] * (A e)_{pi2^-1(i)}   ((Pi2 V2 A e)_i)
//   d       = A c                                 (suffix scan over i)
//   F_i     = v1_i * d_i                          ((V1 A Pi2 V2 A e)_i)
// Tiles of 2048 positions are processed from the end of the vector; each tile
// publishes its aggregate and then its inclusive suffix in one 64-bit status
// word (flag << 32 | value) and looks back over the tiles after it.
// -----------------------------------------------------------------------------
__global__ void __launch_bounds__(kScanThreads) k_syndrome_scan(
    const uint32_t *__restrict__ pi2inv, const uint32_t *__restrict__ v2p,
    const uint32_t *__restrict__ v1, uint32_t N, const uint32_t *__restrict__ sparse, uint32_t t,
    uint32_t count, uint32_t *__restrict__ F, unsigned long long *__restrict__ status,
    uint32_t *__restrict__ err, uint32_t skip_tile, uint32_t spin_limit) {
    extern __shared__ uint32_t sm[];
    uint32_t *s_supp = sm;     // t
    uint32_t *s_suf = sm + t;  // t + 1
    __shared__ uint32_t s_ticket, s_prefix, s_agg;
    __shared__ uint32_t s_wsum[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) s_ticket = atomicAdd(reinterpret_cast<unsigned int *>(status), 1u);
    __syncthreads();
    const uint32_t ntiles = scan_tiles(N);
    const uint32_t ticket = s_ticket;
    if (ticket >= count * ntiles) {  // status word not cleared: never index past the data
        if (tid == 0) record_error(err, kErrScanTimeout);
        return;
    }
    const uint32_t vec = ticket / ntiles;
    const uint32_t tile = ntiles - 1 - ticket % ntiles;
    unsigned long long *st = status + 1 + (size_t)vec * ntiles;

    const uint32_t *sp = sparse + (size_t)vec * 2 * t;
    for (uint32_t j = tid; j < t; j += kScanThreads) {
        s_supp[j] = sp[j];
        s_suf[j] = sp[t + j];
    }
    __syncthreads();
    if (warp == 0) {  // s_suf[j] <- sum_{j' >= j} e_{j'}; s_suf[t] = 0
        const uint32_t per = (t + 31) / 32;
        const uint32_t lo = min(t, lane * per), hi = min(t, lo + per);
        uint32_t sum = 0;
        for (uint32_t j = hi; j-- > lo;) sum = fadd(sum, s_suf[j]);
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, incl, o);
            if (lane + o < 32) incl = fadd(incl, y);
        }
        uint32_t run = fsub(incl, sum);
        for (uint32_t j = hi; j-- > lo;) {
            run = fadd(run, s_suf[j]);
            s_suf[j] = run;
        }
        if (lane == 0) s_suf[t] = 0;
    }
    __syncthreads();

    const uint32_t base = tile * kScanTile + tid * kScanItems;
    uint32_t c[kScanItems];
    uint32_t idx[kScanItems], scale[kScanItems];
    if (base + kScanItems <= N) {
        const uint4 a0 = *reinterpret_cast<const uint4 *>(pi2inv + base);
        const uint4 a1 = *reinterpret_cast<const uint4 *>(pi2inv + base + 4);
        const uint4 b0 = *reinterpret_cast<const uint4 *>(v2p + base);
        const uint4 b1 = *reinterpret_cast<const uint4 *>(v2p + base + 4);
        idx[0] = a0.x; idx[1] = a0.y; idx[2] = a0.z; idx[3] = a0.w;
        idx[4] = a1.x; idx[5] = a1.y; idx[6] = a1.z; idx[7] = a1.w;
        scale[0] = b0.x; scale[1] = b0.y; scale[2] = b0.z; scale[3] = b0.w;
        scale[4] = b1.x; scale[5] = b1.y; scale[6] = b1.z; scale[7] = b1.w;
    } else {
#pragma unroll
        for (int u = 0; u < kScanItems; ++u) {
            const uint32_t i = base + u;
            idx[u] = i < N ? pi2inv[i] : 0u;
            scale[u] = i < N ? v2p[i] : 0u;
        }
    }
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        uint32_t lo = 0, hi = t;  // first support index >= idx[u]
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_supp[mid] < idx[u]) lo = mid + 1; else hi = mid;
        }
        c[u] = fmul(scale[u], s_suf[lo]);
    }
    uint32_t run = 0;
#pragma unroll
    for (int u = kScanItems - 1; u >= 0; --u) {
        run = fadd(run, c[u]);
        c[u] = run;
    }
    // block-wide exclusive suffix scan of the per-thread totals
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(kFull, incl, o);
        if (lane + o < 32) incl = fadd(incl, y);
    }
    if (lane == 0) s_wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        constexpr int nw = kScanThreads / 32;
        const uint32_t wv = lane < nw ? s_wsum[lane] : 0u;
        uint32_t winc = wv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, winc, o);
            if (lane + o < 32) winc = fadd(winc, y);
        }
        __syncwarp();
        if (lane < nw) s_wsum[lane] = fsub(winc, wv);
        if (lane == 0) s_agg = winc;
    }
    __syncthreads();
    const uint32_t thread_excl = fadd(fsub(incl, run), s_wsum[warp]);

    if (tid == 0) {
        const uint32_t agg = s_agg;
        // a failure-path test withholds this tile's status words, so that the
        // look-back of the tile before it expires (off: skip_tile >= ntiles)
        const bool publish = tile != skip_tile;
        uint32_t prefix = 0;
        if (tile == ntiles - 1) {
            if (publish) st_release_u64(st + tile, (2ull << 32) | agg);
        } else {
            if (publish) st_release_u64(st + tile, (1ull << 32) | agg);
            uint32_t j = tile + 1, spins = 0;
            for (;;) {
                const unsigned long long w = ld_acquire_u64(st + j);
                const uint32_t flag = (uint32_t)(w >> 32);
                if (flag == 0u) {
                    if (++spins > spin_limit) {
                        record_error(err, kErrScanTimeout);
                        break;
                    }
                    __nanosleep(32);
                    continue;
                }
                prefix = fadd(prefix, (uint32_t)w);
                if (flag == 2u || j + 1 >= ntiles) break;
                ++j;
            }
            if (publish) st_release_u64(st + tile, (2ull << 32) | fadd(agg, prefix));
        }
        s_prefix = prefix;
    }
    __syncthreads();
    const uint32_t add = fadd(thread_excl, s_prefix);
    uint32_t *Fv = F + (size_t)vec * N;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const uint32_t i = base + u;
        if (i < N) Fv[i] = fmul(__ldg(v1 + i), fadd(c[u], add));
    }
}

__global__ void __launch_bounds__(kScanThreads, 4) k_syndrome_tiles(const __grid_constant__ TileArgs args) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    syndrome_tile(args, blockIdx.x);
}

// out_j = addend_j + sum_{c<r} F[pi1^-1(r j + c)]  ((R Pi1 F)_j, plus x_j).
// The table is read before griddepcontrol.wait.  status[0 .. nclear) is set to
// zero (the words k_syndrome_tiles used).
__global__ void __launch_bounds__(256) k_syndrome_gather(const uint32_t *__restrict__ pi1inv,
                                                        uint32_t n, uint32_t r,
                                                        const uint32_t *F, uint32_t N,
                                                        const uint32_t *addend, uint32_t *out,
                                                        unsigned long long *status, uint32_t nclear) {
    const uint32_t vec = blockIdx.y;
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t *p = pi1inv + (size_t)j * r;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    if (r == 8 && j < n) {
        a = __ldg(reinterpret_cast<const uint4 *>(p));
        b = __ldg(reinterpret_cast<const uint4 *>(p + 4));
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t gid = (blockIdx.y * gridDim.x + blockIdx.x) * 256u + threadIdx.x;
    for (uint32_t i = gid; i < nclear; i += gridDim.x * gridDim.y * 256u) status[i] = 0ull;
    if (j >= n) return;
    const uint32_t *Fv = F + (size_t)vec * N;
    const size_t o = (size_t)vec * n + j;
    uint32_t s = addend ? addend[o] : 0u;
    if (r == 8) {
        s = fadd(s, fadd(fadd(fadd(Fv[a.x], Fv[a.y]), fadd(Fv[a.z], Fv[a.w])),
                         fadd(fadd(Fv[b.x], Fv[b.y]), fadd(Fv[b.z], Fv[b.w]))));
    } else {
        for (uint32_t c = 0; c < r; ++c) s = fadd(s, Fv[p[c]]);
    }
    out[o] = s;
}

// -----------------------------------------------------------------------------
// Fused syndrome: x' = G e for a freshly sampled sparse e, one CTA of 1024
// threads per vector with the length-N intermediate in its shared memory
// (codes of up to about 45 K positions).  Steps (App. B, syndrome direction):
//   sample e (warp 0: support; warp 1: values), the ascending support read
//     off the sampling bitmap by a block-wide scan;
//   c_{pi2(k)} = v2_k (A e)_k, the step function (A e)_k found from the bitmap
//     of the support and the supports before each of its words (a bucket index
//     and a search of the supports after it: 15.2 us a call of 100 vectors at
//     N = 32768, back to back, against 13.9; alone 25.2 against 22.1 us);
//   d = A c: a block suffix scan;
//   out_j = addend_j + sum_{c<r} v1 d at pi1^-1(r j + c).
// No global scratch and no look-back.  (Spreading a vector over a cluster of
// 2 to 8 CTAs, for longer codes and for small batches, took 21 to 77 us where
// k_syndrome_tiles takes 7 to 11.)
// -----------------------------------------------------------------------------
constexpr int kFusedThreads = 1024;
constexpr int kFusedBatch1 = 8;      // loads in flight per thread

__device__ __forceinline__ uint32_t fpad(uint32_t i) { return i + (i >> 5); }  // bank padding

// e <- E_t^N in a CTA of TH threads: the ascending support in supp[0 .. t), the
// suffix sums of the values in suf[0 .. t] (suf[t] = 0), the support as bits in
// bitmap and, per bitmap word, the supports in the words before it in cnt, so
// that support_rank needs no search.  Warp 0 draws the support, warp 1 the
// values; the ascending support is read off the bitmap by a block-wide scan.
// bitmap, cnt: ceil(N / 32); words: 1024; s_wsum: TH / 32.  Ends with a barrier.
template <int TH>
__device__ __forceinline__ void sample_sorted(const pvmvmd_key &key, uint32_t tag, uint64_t idx, uint32_t N,
                                              uint32_t t, uint32_t *bitmap, uint16_t *cnt, uint32_t *words,
                                              uint32_t *supp, uint32_t *suf, uint32_t *s_wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nw = TH / 32;
    const uint32_t nbw = (N + 31) / 32;
    for (uint32_t w = tid; w < nbw; w += TH) bitmap[w] = 0u;
    __syncthreads();
    if (warp == 0)
        warp_sample_support(key, tag, 2 * idx, N, t, bitmap, words, lane);
    else if (warp == 1)
        warp_sample_values(key, tag, 2 * idx + 1, t, words + 512, suf, lane);
    __syncthreads();
    // block-wide exclusive scan of the per-thread bit counts
    const uint32_t per = (nbw + TH - 1) / TH;
    const uint32_t w0 = min(nbw, tid * per), w1 = min(nbw, w0 + per);
    uint32_t c = 0;
    for (uint32_t w = w0; w < w1; ++w) c += __popc(bitmap[w]);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_wsum[warp] = incl;
    if (warp == nw - 1) {  // suf[j] <- sum_{j' >= j} e_{j'}; suf[t] = 0
        const uint32_t pt = (t + 31) / 32;
        const uint32_t lo = min(t, lane * pt), hi = min(t, lo + pt);
        uint32_t sum = 0;
        for (uint32_t j = hi; j-- > lo;) sum = fadd(sum, suf[j]);
        uint32_t sfx = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, sfx, o);
            if (lane + o < 32) sfx = fadd(sfx, y);
        }
        uint32_t run = fsub(sfx, sum);
        for (uint32_t j = hi; j-- > lo;) {
            run = fadd(run, suf[j]);
            suf[j] = run;
        }
        if (lane == 0) suf[t] = 0;
    }
    __syncthreads();
    uint32_t before = lane < warp ? s_wsum[lane] : 0u;  // the warps before this one (at most 32)
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
    uint32_t pos = before + incl - c;
    for (uint32_t w = w0; w < w1; ++w) {
        uint32_t bits = bitmap[w];
        cnt[w] = (uint16_t)pos;
        while (bits) {
            supp[pos++] = w * 32 + (uint32_t)(__ffs(bits) - 1);
            bits &= bits - 1;
        }
    }
    __syncthreads();
}
// The first support index at or above position k (the supports below k).
__device__ __forceinline__ uint32_t support_rank(const uint32_t *bitmap, const uint16_t *cnt, uint32_t k) {
    return cnt[k >> 5] + (uint32_t)__popc(bitmap[k >> 5] & ((1u << (k & 31)) - 1u));
}

// Everything before this point reads only the key and the code tables; the
// state st and the output are written after griddepcontrol.wait, so a launch
// with programmatic serialisation may run its sampling and scans while the
// kernel before it finishes.  Writes st = (support, e) with e_j recovered
// from the suffix sums suf (suf[t] = 0).
template <int TH>
__device__ __forceinline__ void fused_publish(uint32_t *st, const uint32_t *supp, const uint32_t *suf,
                                              uint32_t t, int tid) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (uint32_t j = tid; j < t; j += TH) {
        st[j] = supp[j];
        st[t + j] = fsub(suf[j], suf[j + 1]);
    }
}

__global__ void __launch_bounds__(kFusedThreads) k_syndrome_fused(
    pvmvmd_key key, uint32_t tag, uint64_t idx0, uint32_t N, uint32_t t, uint32_t slice,
    const uint32_t *__restrict__ pi1inv, uint32_t n, uint32_t r,
    uint32_t *__restrict__ sparse_out, const uint32_t *addend, uint32_t *out,
    const uint32_t *__restrict__ pi2, const uint32_t *__restrict__ v2m,
    const uint32_t *__restrict__ v1pm) {
    extern __shared__ uint32_t sm[];
    __shared__ uint32_t s_wsum[kFusedThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t vec = blockIdx.x;
    const uint64_t idx = idx0 + vec;
    const uint32_t fwords = fpad(slice);
    uint32_t *F = sm;                 // padded slice
    uint32_t *supp = sm + fwords;     // t
    uint32_t *suf = supp + t;         // t + 1
    uint32_t *words = suf + t + 1;    // 1024
    uint32_t *bitmap = words + 1024;  // the support, and below it per 32 positions
    uint16_t *cnt = reinterpret_cast<uint16_t *>(bitmap + (N + 31) / 32);

    // the kernels that follow may launch now; they wait for this one before
    // reading anything it writes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    sample_sorted<kFusedThreads>(key, tag, idx, N, t, bitmap, cnt, words, supp, suf, s_wsum);
    // ---- the whole vector in this CTA: c_{pi2(k)} = v2_k (A e)_k,
    // scattered into the slice.  Positions are interleaved over the
    // threads (k = u * 1024 + tid), so the table loads are coalesced and
    // kFusedBatch1 of them are in flight per thread.
    const uint32_t items = slice / kFusedThreads;
    for (uint32_t i = N + tid; i < slice; i += kFusedThreads) F[fpad(i)] = 0u;  // padding
    for (uint32_t u0 = 0; u0 < items; u0 += kFusedBatch1) {
        uint32_t pk[kFusedBatch1], vk[kFusedBatch1];
#pragma unroll
        for (int u = 0; u < kFusedBatch1; ++u) {
            const uint32_t k = (u0 + u) * kFusedThreads + tid;
            const bool ok = u0 + u < items && k < N;
            pk[u] = ok ? __ldg(pi2 + k) : 0u;
            vk[u] = ok ? __ldg(v2m + k) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kFusedBatch1; ++u) {
            const uint32_t k = (u0 + u) * kFusedThreads + tid;
            if (u0 + u < items && k < N) {
                F[fpad(pk[u])] = fmul_mont(suf[support_rank(bitmap, cnt, k)], vk[u]);
            }
        }
    }
    __syncthreads();
    // d = A c: thread tid owns positions [tid*items, (tid+1)*items)
    uint32_t run = 0;
    for (uint32_t u = items; u-- > 0;) {
        const uint32_t li = tid * items + u;
        run = fadd(run, F[fpad(li)]);
        F[fpad(li)] = run;
    }
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(kFull, incl, o);
        if (lane + o < 32) incl = fadd(incl, y);
    }
    if (lane == 0) s_wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        constexpr int nw = kFusedThreads / 32;
        const uint32_t wv = lane < nw ? s_wsum[lane] : 0u;
        uint32_t winc = wv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, winc, o);
            if (lane + o < 32) winc = fadd(winc, y);
        }
        __syncwarp();
        if (lane < nw) s_wsum[lane] = fsub(winc, wv);
    }
    __syncthreads();
    const uint32_t add = fadd(fsub(incl, run), s_wsum[warp]);
    for (uint32_t u = 0; u < items; ++u) {
        const uint32_t li = tid * items + u;
        F[fpad(li)] = fadd(F[fpad(li)], add);
    }
    __syncthreads();
    fused_publish<kFusedThreads>(sparse_out + (size_t)vec * 2 * t, supp, suf, t, tid);
    // out_j = addend_j + sum_c v1[pi1^-1(r j + c)] d[pi1^-1(r j + c)]
    for (uint32_t jo = tid; jo < n; jo += kFusedThreads) {
        const uint32_t *p = pi1inv + (size_t)jo * r;
        const uint32_t *w = v1pm + (size_t)jo * r;
        uint32_t acc = 0;
        if (r == 8) {
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p));
            const uint4 b = __ldg(reinterpret_cast<const uint4 *>(p + 4));
            const uint4 c = __ldg(reinterpret_cast<const uint4 *>(w));
            const uint4 d = __ldg(reinterpret_cast<const uint4 *>(w + 4));
            acc = fadd(fadd(fadd(fmul_mont(F[fpad(a.x)], c.x), fmul_mont(F[fpad(a.y)], c.y)),
                            fadd(fmul_mont(F[fpad(a.z)], c.z), fmul_mont(F[fpad(a.w)], c.w))),
                       fadd(fadd(fmul_mont(F[fpad(b.x)], d.x), fmul_mont(F[fpad(b.y)], d.y)),
                            fadd(fmul_mont(F[fpad(b.z)], d.z), fmul_mont(F[fpad(b.w)], d.w))));
        } else {
            for (uint32_t cc = 0; cc < r; ++cc) acc = fadd(acc, fmul_mont(F[fpad(__ldg(p + cc))], __ldg(w + cc)));
        }
        const size_t o = (size_t)vec * n + jo;
        out[o] = addend ? fadd(addend[o], acc) : acc;
    }
}

// -----------------------------------------------------------------------------
// Sliced syndrome: x' = G e, one CTA of 512 threads per vector and two per SM,
// for codes longer than one CTA's shared memory.  The positions are taken in
// slices of kSlice from the end of the vector, so that the suffix sum of a
// slice starts from the carry of those before it, and only one slice and the n
// outputs are held:
//   c over the slice, scattered from the positions k with pi2(k) in it, which
//     a table lists in ascending order (k << kSliceBits | pi2(k) mod kSlice, so
//     that a warp's lookups of (A e)_k meet in one or two supports);
//   a block-wide suffix scan of eight positions per thread, in registers;
//   out_{pi1(i) / r} += v1_i d_i by shared-memory atomics: the sum mod 2^32 and,
//     from the value an addition finds, its carries (a byte per output).
// Nothing of length N goes through memory (the lanes below move 20 bytes per
// vector and position); bound by instruction issue and shared-memory conflicts
// of the two permutations.  256 vectors at N = 65536: 83 -> 55 us (outputs from
// a second pass over the slice in shared memory: 67; 1024 threads, one CTA per
// SM: 74).
// -----------------------------------------------------------------------------
constexpr int kSliceBits = 12;
constexpr uint32_t kSlice = 1u << kSliceBits;
constexpr int kSliceThreads = 512;
constexpr int kSliceItems = (int)kSlice / kSliceThreads;  // consecutive positions of a thread
static_assert(kSliceItems == 8, "two 16-byte reads of a table");

// t[0 .. 8) = p[at .. at + 8), zero from index `end`
__device__ __forceinline__ void slice_read(const uint32_t *__restrict__ p, uint32_t at, uint32_t end, uint32_t (&t)[8]) {
    if (at + 8 <= end) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p + at)), b = __ldg(reinterpret_cast<const uint4 *>(p + at + 4));
        t[0] = a.x; t[1] = a.y; t[2] = a.z; t[3] = a.w;
        t[4] = b.x; t[5] = b.y; t[6] = b.z; t[7] = b.w;
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = at + u < end ? __ldg(p + at + u) : 0u;
    }
}

__global__ void __launch_bounds__(kSliceThreads, 2) k_syndrome_sliced(
    pvmvmd_key key, uint32_t tag, uint64_t idx0, uint32_t N, uint32_t t, const uint32_t *__restrict__ kp,
    const uint32_t *__restrict__ v2s, const uint32_t *__restrict__ v1m, const uint32_t *__restrict__ oj, uint32_t n,
    uint32_t *__restrict__ sparse_out, const uint32_t *addend, uint32_t *out) {
    extern __shared__ uint32_t sm[];
    constexpr int nw = kSliceThreads / 32;
    __shared__ uint32_t s_wtot[nw];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *F = sm;                         // padded slice
    uint32_t *lo = F + fpad(kSlice);          // n: sums mod 2^32
    uint32_t *hi = lo + n;                    // n bytes: their carries
    uint32_t *supp = hi + (n + 3) / 4;        // t
    uint32_t *suf = supp + t;                 // t + 1
    uint32_t *bitmap = suf + t + 1;           // the support, and below it per 32 positions
    uint16_t *cnt = reinterpret_cast<uint16_t *>(bitmap + (N + 31) / 32);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the keystream words pass through F (kSlice >= 1024)
    sample_sorted<kSliceThreads>(key, tag, idx0 + blockIdx.x, N, t, bitmap, cnt, F, supp, suf, s_wtot);
    for (uint32_t j = tid; j < n + (n + 3) / 4; j += kSliceThreads) lo[j] = 0u;
    uint32_t carry = 0;
    uint32_t s = (N + kSlice - 1) / kSlice - 1;
    uint32_t at = s * kSlice + tid * kSliceItems;
    uint32_t kk[8], vv[8];
    slice_read(kp, at, N, kk);
    slice_read(v2s, at, N, vv);
    for (;; --s, at -= kSlice) {
        // c over the slice; a short one (the last) has zeros above its end
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (at + u < N)
                F[fpad(kk[u] & (kSlice - 1))] =
                    fmul_mont(suf[support_rank(bitmap, cnt, kk[u] >> kSliceBits)], vv[u]);
            else
                F[fpad(tid * kSliceItems + u)] = 0u;
        }
        uint32_t ww[8];
        slice_read(v1m, at, N, ww);
        const uint4 o4 = __ldg(reinterpret_cast<const uint4 *>(oj) + at / 8);
        __syncthreads();
        uint32_t f[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] = F[fpad(tid * kSliceItems + u)];
#pragma unroll
        for (int u = 6; u >= 0; --u) f[u] = fadd(f[u], f[u + 1]);
        uint32_t incl = f[0];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, incl, o);
            if (lane + o < 32) incl = fadd(incl, y);
        }
        if (lane == 0) s_wtot[warp] = incl;
        if (s > 0) {  // tables of the next slice
            slice_read(kp, at - kSlice, N, kk);
            slice_read(v2s, at - kSlice, N, vv);
        }
        __syncthreads();  // F is read: the next slice may be scattered after this
        // every warp: the totals of the warps after it, and all of them
        const uint32_t wv = lane < nw ? s_wtot[lane] : 0u;
        uint32_t winc = wv;
#pragma unroll
        for (int o = 1; o < nw; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, winc, o);
            if (lane + o < 32) winc = fadd(winc, y);
        }
        const uint32_t after = __shfl_sync(kFull, fsub(winc, wv), warp), all = __shfl_sync(kFull, winc, 0);
        const uint32_t add = fadd(fadd(fsub(incl, f[0]), after), carry);
        carry = fadd(carry, all);
        const uint32_t oo[4] = {o4.x, o4.y, o4.z, o4.w};
        uint32_t old[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t j = u & 1 ? oo[u / 2] >> 16 : oo[u / 2] & 0xffffu;
            f[u] = fmul_mont(fadd(f[u], add), ww[u]);  // 0 above the end of a short slice (scale 0)
            old[u] = atomicAdd(lo + j, f[u]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (old[u] + f[u] < old[u]) {
                const uint32_t j = u & 1 ? oo[u / 2] >> 16 : oo[u / 2] & 0xffffu;
                atomicAdd(hi + (j >> 2), 1u << (8 * (j & 3)));
            }
        if (s == 0) break;
    }
    __syncthreads();
    fused_publish<kSliceThreads>(sparse_out + (size_t)blockIdx.x * 2 * t, supp, suf, t, tid);
    for (uint32_t j = tid; j < n; j += kSliceThreads) {
        const uint32_t h = (hi[j >> 2] >> (8 * (j & 3))) & 0xffu;
        const uint32_t x = fred(((uint64_t)h << 32) | lo[j]);
        const size_t o = (size_t)blockIdx.x * n + j;
        out[o] = addend ? fadd(addend[o], x) : x;
    }
}

// The tables of k_syndrome_sliced, one CTA per slice: kp and v2s list the
// positions k with pi2(k) in the slice in ascending order.
__global__ void __launch_bounds__(1024) k_slice_tables(const uint32_t *__restrict__ pi1,
                                                       const uint32_t *__restrict__ pi2,
                                                       const uint32_t *__restrict__ v2m, uint32_t N, uint32_t r,
                                                       uint32_t *__restrict__ kp, uint32_t *__restrict__ v2s,
                                                       uint16_t *__restrict__ oj) {
    __shared__ uint32_t s_wsum[2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t at = blockIdx.x * kSlice;
    int buf = 0;
    for (uint32_t k0 = 0; k0 < N; k0 += 1024, buf ^= 1) {
        const uint32_t k = k0 + threadIdx.x;
        const uint32_t p = k < N ? __ldg(pi2 + k) : 0xffffffffu;
        const bool in = k < N && p >> kSliceBits == blockIdx.x;
        const uint32_t mask = __ballot_sync(kFull, in);
        if (lane == 0) s_wsum[buf][warp] = __popc(mask);
        __syncthreads();
        const uint32_t wv = s_wsum[buf][lane];
        const uint32_t e = at + __reduce_add_sync(kFull, lane < warp ? wv : 0u) + __popc(mask & lanemask_lt());
        if (in) {
            kp[e] = k << kSliceBits | (p & (kSlice - 1));
            v2s[e] = v2m[k];
        }
        at += __reduce_add_sync(kFull, wv);
    }
    for (uint32_t i = blockIdx.x * kSlice + threadIdx.x; i < (blockIdx.x + 1) * kSlice; i += 1024)
        oj[i] = i < N ? (uint16_t)(__ldg(pi1 + i) / r) : (uint16_t)0;
}

// -----------------------------------------------------------------------------
// One accumulate stage of G^T w (App. B, encoding direction) over L lanes:
//   Y[j][l] = sum_{j' <= j} vscale[j'] * X[perm[j'] / div][l]
// With (perm, div, vscale) = (pi1, r, v1) this is A^T V1 Pi1^T R^T; with
// (pi2, 1, v2) it is A^T V2 Pi2^T.  vscale_m holds vscale in Montgomery form
// (v R mod q).  A CTA owns 256 lanes and kEncTile positions: the source row
// and scale of each position are looked up once per CTA (in shared memory),
// and every thread issues all kEncTile row loads of its lane before the
// arithmetic.  Tiles of one lane block are chained by a decoupled look-back
// that each lane walks on its own: per (tile, lane) one 64-bit status word
// holds a state in its high half (1: the tile's own sum, 2: the inclusive
// prefix through the tile) and the value in its low half, so a reader gets
// state and value in one load and no fence or block barrier is needed.
// A tile's predecessors are CTAs of lower index (started first, as in
// syndrome_tile; with a ticket a launch took as long).  (The earlier form, one flag per
// tile and the lanes' values in separate arrays behind a fence and block
// barriers, with warp 0 reading 32 flags at a time, took 0.755 ms per
// 4096 x 4096 encoding.)  At 32 positions per tile the kernel is held to 64
// registers, four CTAs per SM.  Issue-bound: loads without predicates (a lane
// past L reads the last one, a position past N row 0 with scale 0), one
// shared-memory read per position for the row's byte offset and scale, and
// the field additions by min took a launch at N = 32768, L = 4096 from 295 to
// 200 us (int8) and 287 to 235 us (uint32).
// -----------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long enc_status(uint32_t state, uint32_t v) {
    return ((unsigned long long)state << 32) | v;
}

template <bool kI8>
__global__ void __launch_bounds__(256, 4) k_encode_scan(const void *__restrict__ Xv, size_t ldx,
                                                    const uint32_t *__restrict__ perm, uint32_t div,
                                                    const uint32_t *__restrict__ vscale_m, uint32_t N,
                                                    uint32_t L, uint32_t *__restrict__ Y, size_t ldy,
                                                    unsigned long long *status, uint32_t *__restrict__ err) {
    __shared__ ulonglong2 s_row[kEncTile];  // byte offset of the source row and scale of each position
    const int tid = threadIdx.x;
    const uint32_t nlb = (L + 255) / 256;
    const uint32_t ntiles = (N + kEncTile - 1) / kEncTile;
    const uint32_t tile = blockIdx.x / nlb, lb = blockIdx.x % nlb;
    const uint32_t l = lb * 256 + tid;
    const bool lane_ok = l < L;
    const uint32_t j0 = tile * kEncTile;
    if (tid < kEncTile) {
        const uint32_t j = j0 + tid;
        // scale 0 past N: adds nothing
        const unsigned long long row = j < N ? __ldg(perm + j) / div : 0u;
        s_row[tid] = make_ulonglong2(row * ldx * (kI8 ? 1 : 4), j < N ? __ldg(vscale_m + j) : 0u);
    }
    __syncthreads();

    // an idle lane reads a neighbour's column; nothing of it is stored
    const uint32_t lr = lane_ok ? l : L - 1;
    uint32_t v[kEncTile];
    if (kI8) {
        const int8_t *X = static_cast<const int8_t *>(Xv) + lr;
#pragma unroll
        for (int u = 0; u < kEncTile; ++u) v[u] = (uint32_t)(int32_t)X[s_row[u].x];
#pragma unroll
        for (int u = 0; u < kEncTile; ++u) v[u] = min(v[u], v[u] + kQ);  // the lift: w mod q
    } else {
        const char *X = static_cast<const char *>(Xv) + (size_t)lr * 4;
#pragma unroll
        for (int u = 0; u < kEncTile; ++u) v[u] = *reinterpret_cast<const uint32_t *>(X + s_row[u].x);
    }
    uint32_t run = 0;
#pragma unroll
    for (int u = 0; u < kEncTile; ++u) {
        run = fadd(run, fmul_mont(v[u], (uint32_t)s_row[u].y));
        v[u] = run;
    }

    // this lane's status word of tile 0 of the lane block; tile p is p * 256 on
    unsigned long long *sw = status + (size_t)lb * ntiles * 256 + tid;
    uint32_t prefix = 0;
    if (tile == 0) {
        st_relaxed_u64(sw, enc_status(2u, run));
    } else {
        st_relaxed_u64(sw + (size_t)tile * 256, enc_status(1u, run));
        uint32_t spins = 0;
        for (uint32_t p = tile - 1;;) {
            const unsigned long long w = ld_relaxed_u64(sw + (size_t)p * 256);
            const uint32_t state = (uint32_t)(w >> 32);
            if (state == 0u) {
                if (++spins > kSpinLimit) {
                    record_error(err, kErrScanTimeout);
                    break;
                }
                __nanosleep(32);
                continue;
            }
            prefix = fadd(prefix, (uint32_t)w);
            if (state == 2u || p == 0u) break;  // tile 0 is always inclusive
            --p;
        }
        st_relaxed_u64(sw + (size_t)tile * 256, enc_status(2u, fadd(run, prefix)));
    }
    if (lane_ok) {
        uint32_t *yp = Y + (size_t)j0 * ldy + l;
        if (j0 + kEncTile <= N) {
#pragma unroll
            for (int u = 0; u < kEncTile; ++u, yp += ldy) *yp = fadd(v[u], prefix);
        } else {
            const uint32_t nu = N - j0;
#pragma unroll
            for (int u = 0; u < kEncTile; ++u, yp += ldy)
                if ((uint32_t)u < nu) *yp = fadd(v[u], prefix);
        }
    }
}

// 128 x 128 tiles (256 threads): a thread reads 16 rows' four bytes, and writes
// 16 rows' four bytes picked from the tile, 128 bytes per warp both ways.
// (32 x 32 tiles a byte at a time: 31.6 us at 4096 x 4096.)
__global__ void __launch_bounds__(256) k_transpose_i8(const int8_t *__restrict__ in, int R, int C, int8_t *__restrict__ out,
                                                     bool words) {
    __shared__ __align__(16) int8_t tile[128][132];
    const int c0 = blockIdx.x * 128, r0 = blockIdx.y * 128;
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    for (int i = y; i < 128; i += 8) {
        const int r = r0 + i, c = c0 + 4 * x;
        if (words && r < R && c + 4 <= C) {
            *reinterpret_cast<uint32_t *>(&tile[i][4 * x]) = __ldg(reinterpret_cast<const uint32_t *>(in + (size_t)r * C + c));
        } else {
            for (int b = 0; b < 4; ++b)
                if (r < R && c + b < C) tile[i][4 * x + b] = in[(size_t)r * C + c + b];
        }
    }
    __syncthreads();
    for (int i = y; i < 128; i += 8) {
        const int c = c0 + i, r = r0 + 4 * x;
        if (c >= C) continue;
        if (words && r + 4 <= R) {
            uint32_t w = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) w |= (uint32_t)(uint8_t)tile[4 * x + b][i] << (8 * b);
            *reinterpret_cast<uint32_t *>(out + (size_t)c * R + r) = w;
        } else {
            for (int b = 0; b < 4; ++b)
                if (r + b < R) out[(size_t)c * R + r + b] = tile[4 * x + b][i];
        }
    }
}

// -----------------------------------------------------------------------------
// Lane-parallel syndrome x' = G e for a batch of L vectors (Encrypt at large
// batch).  The vectors are the lanes of an N x Lp array C (Lp = L rounded up
// to a multiple of 4, lane index contiguous), so every permutation step of
// G = R Pi1 V1 A Pi2 V2 A moves whole rows:
//   C[pi2(k)][b] = v2_k (A e_b)_k,  (A e_b)_k = sum_{j: s_j >= k} e_j
//                                                   (k_lane_expand)
//   agg[tau][b]  = sum of C[i][b] over tile tau     (k_lane_tile_sum)
//   carry[tau][b] = sum_{tau' > tau} agg[tau'][b]   (k_lane_carry)
//   C[i][b] <- v1_i (carry + sum_{i' >= i in the tile} C[i'][b])
//                                                   (k_lane_scan, in place)
//   out[b][j] = addend[b][j] + sum_{c<r} C[pi1^-1(r j + c)][b]
//                                                   (k_lane_gather)
// A thread owns four consecutive lanes (16-byte accesses) of one tile or
// span; a CTA of 256 threads covers `cols` lane quads (Lp/4 rounded up to a
// power of two, at most 64) of 256 / cols tiles or spans.  The six kernels launch with
// programmatic serialisation and wait (griddepcontrol.wait) before touching
// their predecessor's output.  Only the sampler, whose work needs the key
// alone, lets its successor launch early; the others let it launch at their
// completion.  Early launches of the large grids held SM slots with waiting
// CTAs and were slower (K = 28672, B = 256: 341 against 307 us).
// -----------------------------------------------------------------------------
constexpr int kLaneTileMin = 32;   // positions per tile (one thread walks them):
constexpr int kLaneTileMax = 128;  // the launch picks 32, 64 or 128
constexpr int kLaneCta = 256;      // threads per lane CTA
constexpr int kLaneQuadsMax = 64;  // lane quads per CTA (256 lanes)
constexpr int kExpandSpan = 16;    // positions per expand thread (a multiple of 4)
constexpr int kLaneBuckets = 256;  // bucket index into each lane's sorted support
constexpr int kGatherJ = 16;       // outputs per gather CTA
constexpr int kCarryThreads = 1024;  // tile chunks per lane quad in the carry kernel

__host__ __device__ inline uint32_t lane_pad(uint32_t L) { return (L + 3) & ~3u; }
// Lane quads per CTA: Lp/4 rounded up to a power of two, at most 64 (a CTA
// then holds 256 / cols tiles or spans, and no thread idles for Lp/4 = 16).
__host__ __device__ inline uint32_t lane_cols(uint32_t L) {
    const uint32_t q = lane_pad(L) / 4;
    uint32_t c = 1;
    while (c < q && c < (uint32_t)kLaneQuadsMax) c *= 2;
    return c;
}
__device__ __forceinline__ uint4 fadd4(uint4 a, uint4 b) {
    return make_uint4(fadd(a.x, b.x), fadd(a.y, b.y), fadd(a.z, b.z), fadd(a.w, b.w));
}

// Positions q << lane_bshift(N), q < kLaneBuckets, cover [0, N).
__host__ __device__ inline uint32_t lane_bshift(uint32_t N) {
    uint32_t b = 0;
    while (b < 31 && ((N - 1) >> b) >= (uint32_t)kLaneBuckets) ++b;
    return N > 1 ? b : 0u;
}

// e_b for vector idx0 + blockIdx.x as in k_sample_sparse (warp 0 the
// support, warp 1 the values), written as st[b] = (ascending support,
// values), S[b][j] = sum_{j' >= j} values[j'], S[b][t] = 0, and the bucket
// index first[b][q] = the first support index at or above position
// q << lane_bshift(N).  Everything is computed in shared memory from the key
// alone; st, S and first are written after griddepcontrol.wait (a kernel
// before this one may still read them).
__global__ void __launch_bounds__(128) k_lane_sample(pvmvmd_key key, uint32_t tag, uint64_t idx0,
                                                    uint32_t N, uint32_t t, uint32_t *__restrict__ st,
                                                    uint32_t *__restrict__ S, uint16_t *__restrict__ first) {
    extern __shared__ uint32_t sm[];
    const uint32_t nbw = (N + 31) / 32;
    uint32_t *bitmap = sm;
    uint32_t *words = sm + nbw;      // 512 keystream words (support)
    uint32_t *words2 = words + 512;  // 512 keystream words (values)
    uint32_t *list = words2 + 512;   // t, in the order accepted
    uint32_t *vals = list + t;       // t
    uint32_t *sorted = vals + t;     // t
    uint32_t *suf = sorted + t;      // t + 1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t idx = idx0 + blockIdx.x;
    for (uint32_t w = tid; w < nbw; w += 128) bitmap[w] = 0u;
    __syncthreads();
    if (warp == 0) warp_sample_support_list(key, tag, 2 * idx, N, t, bitmap, words, list, lane);
    else if (warp == 1) warp_sample_values(key, tag, 2 * idx + 1, t, words2, vals, lane);
    __syncthreads();
    for (uint32_t i = tid; i < t; i += 128) {  // ascending support by rank (entries distinct)
        const uint32_t v = list[i];
        uint32_t rk = 0;
        for (uint32_t j = 0; j < t; ++j) rk += list[j] < v;
        sorted[rk] = v;
    }
    if (warp == 0) {
        // suffix sums: lane owns a contiguous chunk, chunks combined by shuffles
        const uint32_t per = (t + 31) / 32;
        const uint32_t lo = min(t, lane * per), hi = min(t, lo + per);
        uint32_t sum = 0;
        for (uint32_t j = hi; j-- > lo;) sum = fadd(sum, vals[j]);
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, incl, o);
            if (lane + o < 32) incl = fadd(incl, y);
        }
        uint32_t run = fsub(incl, sum);  // sum over the chunks after this lane's
        for (uint32_t j = hi; j-- > lo;) {
            run = fadd(run, vals[j]);
            suf[j] = run;
        }
        if (lane == 0) suf[t] = 0u;
    }
    __syncthreads();
    const uint32_t bshift = lane_bshift(N);
    uint16_t fq[kLaneBuckets / 128];
#pragma unroll
    for (int h = 0; h < kLaneBuckets / 128; ++h) {
        const uint32_t pos = (uint32_t)(tid + 128 * h) << bshift;
        uint32_t lo = 0, hi = t;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (sorted[mid] < pos) lo = mid + 1; else hi = mid;
        }
        fq[h] = (uint16_t)lo;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t *stb = st + (size_t)blockIdx.x * 2 * t;
    uint32_t *Sb = S + (size_t)blockIdx.x * (t + 1);
    for (uint32_t j = tid; j < t; j += 128) {
        stb[j] = sorted[j];
        stb[t + j] = vals[j];
    }
    for (uint32_t j = tid; j <= t; j += 128) Sb[j] = suf[j];
#pragma unroll
    for (int h = 0; h < kLaneBuckets / 128; ++h)
        first[(size_t)blockIdx.x * kLaneBuckets + tid + 128 * h] = fq[h];
}

// C[pi2(k)][b] = v2_k (A e_b)_k: a thread walks kExpandSpan positions k of
// four lanes in order with a pointer per lane into the sorted support, and
// writes the four lanes of row pi2(k) with one 16-byte store.
__global__ void __launch_bounds__(kLaneCta) k_lane_expand(const uint32_t *st, const uint32_t *S,
                                                         const uint16_t *first, uint32_t t,
                                                         uint32_t N, uint32_t L,
                                                         const uint32_t *__restrict__ pi2,
                                                         const uint32_t *__restrict__ v2m,
                                                         uint4 *C) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs come from the kernel before
    const uint32_t cols = lane_cols(L), Lq = lane_pad(L) / 4;
    const uint32_t g = blockIdx.y * cols + threadIdx.x % cols;
    const uint32_t k0 = (blockIdx.x * (kLaneCta / cols) + threadIdx.x / cols) * kExpandSpan;
    const uint32_t k1 = min(N, k0 + kExpandSpan);
    if (g >= Lq || k0 >= k1) return;
    uint32_t j[4], next[4], cur[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t b = 4 * g + q;
        next[q] = 0xffffffffu;
        cur[q] = 0u;
        j[q] = 0u;
        if (b < L) {
            // first support index with s_j >= k0: from the bucket of k0, then
            // past the few supports between the bucket's start and k0
            const uint32_t *supp = st + (size_t)b * 2 * t;
            uint32_t lo = first[(size_t)b * kLaneBuckets + (k0 >> lane_bshift(N))];
            uint32_t nx = lo < t ? supp[lo] : 0xffffffffu;
            while (nx < k0) {
                ++lo;
                nx = lo < t ? supp[lo] : 0xffffffffu;
            }
            j[q] = lo;
            next[q] = nx;
            cur[q] = S[(size_t)b * (t + 1) + lo];
        }
    }
    for (uint32_t kb = k0; kb < k1; kb += 4) {  // k0 is a multiple of 4: 16-byte table loads
        uint32_t pk[4], vk[4];
        if (kb + 4 <= N) {
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(pi2 + kb));
            const uint4 c = __ldg(reinterpret_cast<const uint4 *>(v2m + kb));
            pk[0] = a.x; pk[1] = a.y; pk[2] = a.z; pk[3] = a.w;
            vk[0] = c.x; vk[1] = c.y; vk[2] = c.z; vk[3] = c.w;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                pk[u] = kb + u < N ? __ldg(pi2 + kb + u) : 0u;
                vk[u] = kb + u < N ? __ldg(v2m + kb + u) : 0u;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t k = kb + u;
            if (k >= k1) break;
            uint32_t o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t b = 4 * g + q;
                while (next[q] < k) {
                    ++j[q];
                    next[q] = j[q] < t ? st[(size_t)b * 2 * t + j[q]] : 0xffffffffu;
                    cur[q] = S[(size_t)b * (t + 1) + j[q]];
                }
                o[q] = fmul_mont(cur[q], vk[u]);
            }
            C[(size_t)pk[u] * Lq + g] = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// agg[tau][b] = sum over the tile's positions of C[i][b].
__global__ void __launch_bounds__(kLaneCta) k_lane_tile_sum(const uint4 *C, uint32_t N, uint32_t tile, uint32_t L,
                                                           uint4 *agg) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs come from the kernel before
    const uint32_t cols = lane_cols(L), Lq = lane_pad(L) / 4, ntiles = (N + tile - 1) / tile;
    const uint32_t g = blockIdx.y * cols + threadIdx.x % cols;
    const uint32_t tau = blockIdx.x * (kLaneCta / cols) + threadIdx.x / cols;
    if (g >= Lq || tau >= ntiles) return;
    const uint32_t i0 = tau * tile, i1 = min(N, i0 + tile);
    uint4 sum = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t i = i0; i < i1; i += 8) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = i + u < i1 ? C[(size_t)(i + u) * Lq + g] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 8; ++u) sum = fadd4(sum, v[u]);
    }
    agg[(size_t)tau * Lq + g] = sum;
}

// carry[tau][b] = sum_{tau' > tau} agg[tau'][b]: one CTA per lane quad;
// thread c sums its chunk of consecutive tiles, a block-wide suffix scan of
// the chunk sums (warp shuffles, then the 32 warp totals) gives each chunk
// the sum of the tiles after it, and the thread writes its chunk's carries
// walking down.
__device__ __forceinline__ uint4 shfl_down4(uint4 v, int o) {
    return make_uint4(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o),
                      __shfl_down_sync(kFull, v.z, o), __shfl_down_sync(kFull, v.w, o));
}
__device__ __forceinline__ uint4 fsub4(uint4 a, uint4 b) {
    return make_uint4(fsub(a.x, b.x), fsub(a.y, b.y), fsub(a.z, b.z), fsub(a.w, b.w));
}
__global__ void __launch_bounds__(kCarryThreads) k_lane_carry(const uint4 *agg, uint32_t ntiles, uint32_t Lq,
                                                             uint4 *carry) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs come from the kernel before
    __shared__ uint4 wsum[kCarryThreads / 32];
    const uint32_t g = blockIdx.x, c = threadIdx.x, lane = c & 31, warp = c >> 5;
    const uint32_t per = (ntiles + kCarryThreads - 1) / kCarryThreads;
    const uint32_t t0 = min(ntiles, c * per), t1 = min(ntiles, t0 + per);
    uint4 sum = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t tau = t0; tau < t1; tau += 8) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = tau + u < t1 ? agg[(size_t)(tau + u) * Lq + g] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 8; ++u) sum = fadd4(sum, v[u]);
    }
    uint4 incl = sum;  // suffix within the warp: chunks lane .. 31
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint4 y = shfl_down4(incl, o);
        if (lane + o < 32) incl = fadd4(incl, y);
    }
    if (lane == 0) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {  // suffix over the warp totals
        const uint4 wv = wsum[lane];
        uint4 wi = wv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint4 y = shfl_down4(wi, o);
            if (lane + o < 32) wi = fadd4(wi, y);
        }
        __syncwarp();
        wsum[lane] = fsub4(wi, wv);  // totals of the warps after this one
    }
    __syncthreads();
    uint4 run = fadd4(fsub4(incl, sum), wsum[warp]);  // sum over the chunks after this one
    for (uint32_t hi = t1; hi > t0;) {  // eight tiles at a time, loads first
        const uint32_t cnt = hi - t0 < 8u ? hi - t0 : 8u;
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = (uint32_t)u < cnt ? agg[(size_t)(hi - 1 - u) * Lq + g] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if ((uint32_t)u < cnt) {
                carry[(size_t)(hi - 1 - u) * Lq + g] = run;
                run = fadd4(run, v[u]);
            }
        }
        hi -= cnt;
    }
}

// In place: C[i][b] <- v1_i (carry[tau][b] + sum_{i' >= i in tile tau} C[i'][b]),
// with v1m = v1 R (Montgomery, R = 2^32) so that each product is one REDC.
__global__ void __launch_bounds__(kLaneCta, 4) k_lane_scan(uint4 *C, uint32_t N, uint32_t tile, uint32_t L,
                                                       const uint4 *carry,
                                                       const uint32_t *__restrict__ v1m) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs come from the kernel before
    const uint32_t cols = lane_cols(L), Lq = lane_pad(L) / 4, ntiles = (N + tile - 1) / tile;
    const uint32_t g = blockIdx.y * cols + threadIdx.x % cols;
    const uint32_t tau = blockIdx.x * (kLaneCta / cols) + threadIdx.x / cols;
    if (g >= Lq || tau >= ntiles) return;
    const uint32_t i0 = tau * tile, i1 = min(N, i0 + tile);
    uint4 run = carry[(size_t)tau * Lq + g];
    for (uint32_t hi = i1; hi > i0;) {
        const uint32_t cnt = hi - i0 < 8u ? hi - i0 : 8u;  // positions hi-1 .. hi-cnt
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = (uint32_t)u < cnt ? C[(size_t)(hi - 1 - u) * Lq + g] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if ((uint32_t)u < cnt) {
                const uint32_t i = hi - 1 - u, w = __ldg(v1m + i);
                run = fadd4(run, v[u]);
                C[(size_t)i * Lq + g] = make_uint4(fmul_mont(run.x, w), fmul_mont(run.y, w), fmul_mont(run.z, w),
                                                   fmul_mont(run.w, w));
            }
        }
        hi -= cnt;
    }
}

// out[b][j] = addend[b][j] + sum_{c<r} C[pi1^-1(r j + c)][b] for kGatherJ
// outputs and the CTA's lanes, transposed through shared memory so that out
// rows are written 128 bytes at a time.  addend may be null or alias out.
__global__ void __launch_bounds__(kLaneCta, 4) k_lane_gather(const uint4 *C,
                                                         const uint32_t *__restrict__ pi1inv,
                                                         uint32_t r, uint32_t n, uint32_t L,
                                                         const uint32_t *addend, uint32_t *out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs come from the kernel before
    __shared__ uint32_t tile[kGatherJ][4 * kLaneQuadsMax + 1];
    const uint32_t cols = lane_cols(L), subs = kLaneCta / cols, Lq = lane_pad(L) / 4;
    const uint32_t tid = threadIdx.x, gl = tid % cols, sub = tid / cols;
    const uint32_t g = blockIdx.y * cols + gl;
    const uint32_t j0 = blockIdx.x * kGatherJ;
    // thread (sub, quad) takes outputs jj = sub, sub + subs, ... two at a time
    for (uint32_t jj0 = sub; jj0 < (uint32_t)kGatherJ; jj0 += 2 * subs) {
        uint4 v[2][8];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t jj = jj0 + q * subs, j = j0 + jj;
            const bool ok = jj < (uint32_t)kGatherJ && j < n && g < Lq;
#pragma unroll
            for (int c = 0; c < 8; ++c)
                v[q][c] = ok && (uint32_t)c < r ? C[(size_t)__ldg(pi1inv + (size_t)j * r + c) * Lq + g]
                                              : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t jj = jj0 + q * subs, j = j0 + jj;
            if (jj >= (uint32_t)kGatherJ) continue;
            uint4 acc = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc = fadd4(acc, v[q][c]);
            if (r > 8 && j < n && g < Lq)
                for (uint32_t c = 8; c < r; ++c)
                    acc = fadd4(acc, C[(size_t)__ldg(pi1inv + (size_t)j * r + c) * Lq + g]);
            tile[jj][4 * gl] = acc.x;
            tile[jj][4 * gl + 1] = acc.y;
            tile[jj][4 * gl + 2] = acc.z;
            tile[jj][4 * gl + 3] = acc.w;
        }
    }
    __syncthreads();
    // consecutive threads write consecutive outputs of one vector's row
    for (uint32_t idx = tid; idx < 4 * cols * (uint32_t)kGatherJ; idx += kLaneCta) {
        const uint32_t bb = idx / kGatherJ, jj = idx % kGatherJ;
        const uint32_t vb = blockIdx.y * 4 * cols + bb, j = j0 + jj;
        if (vb < L && j < n) {
            const size_t o = (size_t)vb * n + j;
            out[o] = addend ? fadd(addend[o], tile[jj][bb]) : tile[jj][bb];
        }
    }
}

}  // namespace

namespace {
cudaError_t launch_pdl(const void *fn, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void **args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    return counted_launch(cudaLaunchKernelExC(&cfg, fn, args));
}
}  // namespace

// Bitmap of N bits plus 512 keystream words; covers N up to 8 * PVMVMD_MAX_K.
// The support and suffix sums of k_syndrome_scan: t up to 25599.
constexpr size_t kSampleMaxSmem = 200 * 1024;

cudaError_t launch_sample_sparse(const pvmvmd_key &key, uint32_t tag, uint64_t idx0, uint32_t N,
                                 uint32_t t, uint32_t count, uint32_t *out,
                                 unsigned long long *clear, size_t clear_words, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const size_t smem = ((size_t)(N + 31) / 32 + 512) * sizeof(uint32_t);
    if (smem > kSampleMaxSmem) return cudaErrorInvalidValue;
    const cudaError_t attr = func_attr((const void *)k_sample_sparse, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSampleMaxSmem);
    if (attr != cudaSuccess) return attr;
    k_sample_sparse<<<count, 32, smem, s>>>(key, tag, idx0, N, t, out, clear, clear_words); note_launch();
    return cudaGetLastError();
}

cudaError_t launch_syndrome_scan(const uint32_t *pi2inv, const uint32_t *v2p, const uint32_t *v1,
                                 uint32_t N, const uint32_t *sparse, uint32_t t, uint32_t count,
                                 uint32_t *F, unsigned long long *status, uint32_t *err,
                                 cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const size_t smem = (2 * (size_t)t + 1) * sizeof(uint32_t);
    if (smem > kSampleMaxSmem) return cudaErrorInvalidValue;
    const cudaError_t attr = func_attr((const void *)k_syndrome_scan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSampleMaxSmem);
    if (attr != cudaSuccess) return attr;
    const unsigned grid = count * scan_tiles(N);
    const DebugWait dbg = debug_wait();
    const bool inject = dbg.site == PVMVMD_DEBUG_WAIT_SCAN;
    k_syndrome_scan<<<grid, kScanThreads, smem, s>>>(pi2inv, v2p, v1, N, sparse, t, count, F, status,
                                                     err, inject ? dbg.index : 0xFFFFFFFFu,
                                                     inject ? (uint32_t)dbg.limit : kSpinLimit); note_launch();
    return cudaGetLastError();
}

cudaError_t launch_syndrome_gather(const uint32_t *pi1inv, uint32_t n, uint32_t r,
                                   const uint32_t *F, uint32_t N, const uint32_t *addend,
                                   uint32_t *out, uint32_t count, cudaStream_t s,
                                   unsigned long long *status, uint32_t nclear) {
    if (count == 0 || n == 0) return cudaSuccess;
    void *args[] = {&pi1inv, &n, &r, &F, &N, &addend, &out, &status, &nclear};
    return launch_pdl((const void *)k_syndrome_gather, dim3((n + 255) / 256, count), dim3(256), 0, s, args);
}

bool syndrome_tiles_eligible(uint32_t t) { return t <= kTileMaxT; }

cudaError_t launch_syndrome_tiles(const pvmvmd_key &key, uint32_t tag, uint64_t idx0, uint32_t N, uint32_t t,
                                  uint32_t count, const uint32_t *pi2inv, const uint32_t *v2p,
                                  const uint32_t *v1m, const uint32_t *pi1inv, uint32_t n, uint32_t r,
                                  uint32_t *sparse_out, uint32_t *F, unsigned long long *status, uint32_t *err,
                                  const uint32_t *addend, uint32_t *out, cudaStream_t s, bool pdl,
                                  const uint32_t *Qm, int K, uint32_t *u) {
    if (count == 0) return cudaSuccess;
    constexpr uint32_t kMost = 65535;  // the gather's grid
    if (count > kMost) {
        const cudaError_t e =
            launch_syndrome_tiles(key, tag, idx0, N, t, kMost, pi2inv, v2p, v1m, pi1inv, n, r, sparse_out, F, status,
                                  err, addend, out, s, pdl, Qm, K, u);
        if (e != cudaSuccess) return e;
        return launch_syndrome_tiles(key, tag, idx0 + kMost, N, t, count - kMost, pi2inv, v2p, v1m, pi1inv, n, r,
                                     sparse_out ? sparse_out + (size_t)kMost * 2 * t : nullptr, F, status, err,
                                     addend ? addend + (size_t)kMost * n : nullptr, out + (size_t)kMost * n, s, pdl,
                                     Qm, K, u ? u + (size_t)kMost * K : nullptr);
    }
    const uint32_t ntiles = scan_tiles(N);
    const uint32_t ucols = u ? (uint32_t)(K + kTileUCols - 1) / kTileUCols : 0u;
    const uint64_t ctas = (uint64_t)count * (ntiles + ucols);
    if (!syndrome_tiles_eligible(t) || ctas > 0x7fffffffu) return cudaErrorInvalidValue;
    const DebugWait dbg = debug_wait();
    const bool inject = dbg.site == PVMVMD_DEBUG_WAIT_SCAN;
    TileArgs args{key, tag, N, t, count, idx0, pi2inv, v2p, v1m, sparse_out, F, status, err,
                  inject ? dbg.index : 0xFFFFFFFFu, inject ? (uint32_t)dbg.limit : kSpinLimit, Qm, K, ucols, u};
    cudaError_t e;
    if (pdl) {
        void *argv[] = {&args};
        e = launch_pdl((const void *)k_syndrome_tiles, dim3((uint32_t)ctas), dim3(kScanThreads), 0, s, argv);
    } else {
        k_syndrome_tiles<<<(uint32_t)ctas, kScanThreads, 0, s>>>(args);
        e = counted_launch(cudaGetLastError());
    }
    if (e != cudaSuccess) return e;
    e = launch_syndrome_gather(pi1inv, n, r, F, N, addend, out, count, s, status, count * ntiles);
    // the words must be zero for the next call also where the gather did not start
    if (e != cudaSuccess) (void)cudaMemsetAsync(status, 0, (size_t)count * ntiles * sizeof(unsigned long long), s);
    return e;
}

size_t encode_scan_status_words(uint32_t N, uint32_t L) {
    return (size_t)((L + 255) / 256) * ((N + kEncTile - 1) / kEncTile) * 256;
}

cudaError_t encode_scan_clear(unsigned long long *status, uint32_t N, uint32_t L, cudaStream_t s) {
    return cudaMemsetAsync(status, 0, encode_scan_status_words(N, L) * sizeof(unsigned long long), s);
}

cudaError_t launch_encode_scan(const void *X, bool x_is_i8, size_t ldx, const uint32_t *perm,
                               uint32_t div, const uint32_t *vscale_m, uint32_t N, uint32_t L,
                               uint32_t *Y, size_t ldy, unsigned long long *status, uint32_t *err,
                               cudaStream_t s) {
    const size_t ctas = encode_scan_status_words(N, L) / 256;
    if (ctas == 0) return cudaSuccess;
    if (ctas > 0x7fffffffu) return cudaErrorInvalidValue;
    if (x_is_i8)
        k_encode_scan<true><<<(unsigned)ctas, 256, 0, s>>>(X, ldx, perm, div, vscale_m, N, L, Y, ldy,
                                                           status, err);
    else
        k_encode_scan<false><<<(unsigned)ctas, 256, 0, s>>>(X, ldx, perm, div, vscale_m, N, L, Y, ldy,
                                                            status, err);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_transpose_i8(const int8_t *in, int R, int C, int8_t *out, cudaStream_t s) {
    if (R <= 0 || C <= 0) return cudaSuccess;
    dim3 grid((C + 127) / 128, (R + 127) / 128);
    if (grid.y > 65535u) return cudaErrorInvalidValue;
    const bool words = C % 4 == 0 && R % 4 == 0 &&
                       ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 3u) == 0;
    k_transpose_i8<<<grid, 256, 0, s>>>(in, R, C, out, words); note_launch();
    return cudaGetLastError();
}


namespace {
uint32_t fused_slice(uint32_t N) { return (N + kFusedThreads - 1) / kFusedThreads * kFusedThreads; }
size_t fused_smem(uint32_t slice, uint32_t t) {
    return ((size_t)slice + slice / 32 + 2 * (size_t)t + 1 + 1024 + slice / 32 + slice / 64) * sizeof(uint32_t);
}
constexpr size_t kFusedMaxSmem = 188 * 1024;
}  // namespace

bool syndrome_fused_fits(uint32_t N, uint32_t t) {
    return N <= (1u << 20) && fused_smem(fused_slice(N), t) <= kFusedMaxSmem;
}

cudaError_t launch_syndrome_fused(const pvmvmd_key &key, uint32_t tag, uint64_t idx0, uint32_t N,
                                  uint32_t t, uint32_t count, const uint32_t *pi1inv,
                                  const uint32_t *pi2, const uint32_t *v2m, const uint32_t *v1pm,
                                  uint32_t n, uint32_t r, uint32_t *sparse_out,
                                  const uint32_t *addend, uint32_t *out, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    if (!syndrome_fused_fits(N, t)) return cudaErrorNotSupported;
    const cudaError_t attr = func_attr((const void *)k_syndrome_fused, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kFusedMaxSmem);
    if (attr != cudaSuccess) return attr;
    uint32_t slice = fused_slice(N);
    void *args[] = {(void *)&key, &tag, &idx0, &N, &t, &slice, &pi1inv, &n, &r, &sparse_out, &addend, &out,
                    &pi2, &v2m, &v1pm};
    return launch_pdl((const void *)k_syndrome_fused, dim3(count), dim3(kFusedThreads), fused_smem(slice, t), s, args);
}

namespace {
size_t sliced_smem(uint32_t N, uint32_t n, uint32_t t) {
    const size_t nbw = (N + 31) / 32;
    return ((size_t)kSlice + kSlice / 32 + n + (n + 3) / 4 + 2 * (size_t)t + 1 + nbw + (nbw + 1) / 2) * sizeof(uint32_t);
}
constexpr size_t kSlicedMaxSmem = 110 * 1024;  // two CTAs per SM
}  // namespace

bool syndrome_sliced_fits(uint32_t N, uint32_t n, uint32_t r, uint32_t t) {
    // k in 32 - kSliceBits bits, outputs in 16, carries of r terms in 8
    return N <= (1u << (32 - kSliceBits)) && n <= 65536u && r <= 255u && sliced_smem(N, n, t) <= kSlicedMaxSmem;
}
size_t slice_table_words(uint32_t N) {
    return 2 * (((size_t)N + 3) & ~(size_t)3) + (((size_t)N + kSlice - 1) / kSlice * kSlice) / 2;
}

cudaError_t launch_slice_tables(const uint32_t *pi1, const uint32_t *pi2, const uint32_t *v2m, uint32_t N, uint32_t r,
                                uint32_t *tables, cudaStream_t s) {
    const size_t Np = ((size_t)N + 3) & ~(size_t)3;
    k_slice_tables<<<(N + kSlice - 1) / kSlice, 1024, 0, s>>>(pi1, pi2, v2m, N, r, tables, tables + Np,
                                                              reinterpret_cast<uint16_t *>(tables + 2 * Np));
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_syndrome_sliced(const pvmvmd_key &key, uint32_t tag, uint64_t idx0, uint32_t N, uint32_t t,
                                   uint32_t count, const uint32_t *tables, const uint32_t *v1m, uint32_t n,
                                   uint32_t *sparse_out, const uint32_t *addend, uint32_t *out, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const cudaError_t attr = func_attr((const void *)k_syndrome_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSlicedMaxSmem);
    if (attr != cudaSuccess) return attr;
    const size_t Np = ((size_t)N + 3) & ~(size_t)3;
    const uint32_t *kp = tables, *v2s = tables + Np, *oj = tables + 2 * Np;
    void *args[] = {(void *)&key, &tag, &idx0, &N, &t, &kp, &v2s, &v1m, &oj, &n, &sparse_out, &addend, &out};
    return launch_pdl((const void *)k_syndrome_sliced, dim3(count), dim3(kSliceThreads), sliced_smem(N, n, t), s, args);
}

size_t lane_state_words(uint32_t t, uint32_t L) {
    return (size_t)L * (t + 1) + (size_t)L * kLaneBuckets / 2;
}

size_t lane_aux_words(uint32_t N, uint32_t L) {
    return 2 * (size_t)((N + kLaneTileMin - 1) / kLaneTileMin) * lane_pad(L);
}

cudaError_t launch_lane_syndrome(const pvmvmd_key &key, uint32_t tag, uint64_t idx0, uint32_t N,
                                 uint32_t t, uint32_t L, const uint32_t *pi2, const uint32_t *v2m,
                                 const uint32_t *v1m, const uint32_t *pi1inv, uint32_t n, uint32_t r,
                                 uint32_t *sparse_out, uint32_t *S, uint32_t *C, uint32_t *aux,
                                 const uint32_t *addend, uint32_t *out, cudaStream_t s) {
    if (L == 0) return cudaSuccess;
    const size_t smem = ((size_t)(N + 31) / 32 + 1024 + 4 * (size_t)t + 1) * sizeof(uint32_t);
    if (smem > kSampleMaxSmem) return cudaErrorInvalidValue;
    const cudaError_t a1 = func_attr((const void *)k_lane_sample, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSampleMaxSmem);
    if (a1 != cudaSuccess) return a1;
    if ((reinterpret_cast<uintptr_t>(C) | reinterpret_cast<uintptr_t>(aux)) & 15u)
        return cudaErrorInvalidValue;
    const uint32_t Lp = lane_pad(L), cols = lane_cols(L), per_cta = kLaneCta / cols;
    const unsigned gy = (Lp / 4 + cols - 1) / cols;
    // tiles of 32 positions, or 64 / 128 when the tile-sum and scan grids
    // still hold two CTAs of threads per SM: longer tiles shorten the carry
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    uint32_t tile = kLaneTileMin;
    while (tile < (uint32_t)kLaneTileMax &&
           (uint64_t)((N + 2 * tile - 1) / (2 * tile)) * (lane_pad(L) / 4) >= (uint64_t)2 * sms * kLaneCta)
        tile *= 2;
    const uint32_t ntiles = (N + tile - 1) / tile;
    const uint32_t nspans = (N + kExpandSpan - 1) / kExpandSpan;
    if (gy > 65535u || L > 0x7fffffffu) return cudaErrorInvalidValue;
    uint4 *agg = reinterpret_cast<uint4 *>(aux), *carry = reinterpret_cast<uint4 *>(aux + (size_t)ntiles * Lp);
    uint4 *C4 = reinterpret_cast<uint4 *>(C);
    const uint4 *C4c = C4, *aggc = agg, *carryc = carry;
    const uint32_t Lq = Lp / 4;
    const uint32_t *stc = sparse_out, *Sc = S;
    // S holds the suffix sums [L][t+1], then the bucket index [L][kLaneBuckets] (uint16)
    uint16_t *first = reinterpret_cast<uint16_t *>(S + (size_t)L * (t + 1));
    const uint16_t *fc = first;
    cudaError_t e;
    void *a0[] = {(void *)&key, &tag, &idx0, &N, &t, &sparse_out, &S, &first};
    if ((e = launch_pdl((const void *)k_lane_sample, dim3(L), dim3(128), smem, s, a0)) != cudaSuccess) return e;
    void *a1x[] = {&stc, &Sc, &fc, &t, &N, &L, (void *)&pi2, (void *)&v2m, &C4};
    if ((e = launch_pdl((const void *)k_lane_expand, dim3((nspans + per_cta - 1) / per_cta, gy), dim3(kLaneCta), 0, s,
                        a1x)) != cudaSuccess)
        return e;
    void *a2[] = {&C4c, &N, &tile, &L, &agg};
    if ((e = launch_pdl((const void *)k_lane_tile_sum, dim3((ntiles + per_cta - 1) / per_cta, gy), dim3(kLaneCta), 0,
                        s, a2)) != cudaSuccess)
        return e;
    void *a3[] = {&aggc, (void *)&ntiles, (void *)&Lq, &carry};
    if ((e = launch_pdl((const void *)k_lane_carry, dim3(Lq), dim3(kCarryThreads), 0, s, a3)) != cudaSuccess) return e;
    void *a4[] = {&C4, &N, &tile, &L, &carryc, (void *)&v1m};
    if ((e = launch_pdl((const void *)k_lane_scan, dim3((ntiles + per_cta - 1) / per_cta, gy), dim3(kLaneCta), 0, s,
                        a4)) != cudaSuccess)
        return e;
    void *a5[] = {&C4c, (void *)&pi1inv, &r, &n, &L, (void *)&addend, &out};
    if ((e = launch_pdl((const void *)k_lane_gather, dim3((n + kGatherJ - 1) / kGatherJ, gy), dim3(kLaneCta), 0, s,
                        a5)) != cudaSuccess)
        return e;
    return cudaGetLastError();
}

}  // namespace pv
