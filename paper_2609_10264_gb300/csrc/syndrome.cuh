// Device code of the tiled syndrome, shared by the kernel of its own (raa.cu)
// and the decode kernel (decode.cu): the samplers of a CTA that draws e itself,
// and one CTA's tile.
#pragma once

#include "common.cuh"
#include "launch.h"

namespace pv {
namespace {

__device__ __forceinline__ int bitlen32(uint32_t v) { return v ? 32 - __clz(v) : 0; }

// Warp: the support of e <- E_t^N in the order accepted -> list[0..t), for
// t <= kTileMaxT without a bitmap: a draw is compared with the list itself
// (16 bytes per shared-memory read, every lane the same address).  list is
// 16-byte aligned and holds kTileMaxT words.
constexpr uint32_t kTileMaxT = 512;
__device__ void warp_sample_support_short(const pvmvmd_key &key, uint32_t tag, uint64_t sidx, uint32_t N,
                                          uint32_t t, uint32_t *words, uint32_t *list, int lane) {
    // unused slots hold a value no draw takes (draws are below N)
    for (uint32_t i = lane; i < ((t + 3) & ~3u); i += 32) list[i] = 0xffffffffu;
    __syncwarp();
    if (N <= 1) {
        if (lane == 0) list[0] = 0u;
        __syncwarp();
        return;
    }
    const int shift = 32 - bitlen32(N - 1);
    uint32_t have = 0;
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
            bool seen = false;
            for (uint32_t h = 0; h < have; h += 4) {
                const uint4 a = *reinterpret_cast<const uint4 *>(list + h);
                seen |= (a.x == v) | (a.y == v) | (a.z == v) | (a.w == v);
            }
            const uint32_t vmask = __ballot_sync(kFull, valid);
            const uint32_t same = __match_any_sync(kFull, valid ? v : 0xffffffffu);
            const bool cand = valid && !seen && (same & vmask & lanemask_lt()) == 0u;
            const uint32_t cmask = __ballot_sync(kFull, cand);
            const uint32_t need = t - have, rk = __popc(cmask & lanemask_lt());
            if (cand && rk < need) list[have + rk] = v;
            have += min((uint32_t)__popc(cmask), need);
            __syncwarp();
        }
        __syncwarp();
    }
}

// Warp: the first t draws of F* from stream (tag, vidx) -> dst.
__device__ void warp_sample_values(const pvmvmd_key &key, uint32_t tag, uint64_t vidx, uint32_t t,
                                   uint32_t *words, uint32_t *dst, int lane) {
    uint32_t have = 0;
    for (uint64_t wpos = 0; have < t; wpos += 512) {
        uint32_t blk[16];
        chacha20_block_dev(key, (uint32_t)(wpos / 16 + lane), tag, (uint32_t)vidx,
                           (uint32_t)(vidx >> 32), blk);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 16; ++i) words[lane * 16 + i] = blk[i];
        __syncwarp();
        for (int batch = 0; batch < 16 && have < t; ++batch) {
            const uint32_t v = words[batch * 32 + lane] >> 1;
            const bool valid = v != 0u && v < kQ;
            const uint32_t m = __ballot_sync(kFull, valid);
            const uint32_t r = __popc(m & lanemask_lt());
            if (valid && have + r < t) dst[have + r] = v;
            have = min(have + (uint32_t)__popc(m), t);
        }
    }
    __syncwarp();
}

// -----------------------------------------------------------------------------
// Tiled syndrome, first half, for `count` freshly sampled sparse vectors:
// every CTA of 256 threads takes one tile of kScanTile positions of one vector
// and draws that vector's e itself (a draw costs about 2 us of latency and no
// traffic), so one launch holds as many small CTAs as there are tiles; they
// fit beside a decrypt's.  The tables of a tile are requested before the
// draw.  Tile sums are chained by a look-back over the tiles after it: their
// own sums only, 32 at a time by one warp, since all of them are published
// at about the same time.  A tile waits only for CTAs of lower index: GPUs start
// blocks in that order, though CUDA does not promise it, and where one did
// not, the bounded waits would run out and be reported (a ticket per CTA would
// cost each call an atomic's latency).  status holds one 64-bit word per (vector, tile)
// (1 << 32 | sum), zero at launch; the gather kernel that follows clears it.
//
// Latency-bound.  Against one cluster of 2 to 8 CTAs of 1024 threads per
// vector (and e^T Q in a kernel after it): decode of 14336 x 4096, 64 vectors
// 115.1 -> 101.6 us, of 4096 x 4096, 100 vectors 55.9 -> 49.4 us; round trip of
// 4096 x 2560, 8 vectors, 16-bit weights 91.7 -> 67.8 us; a mask alone, 8
// vectors: K = 8192 43.1 -> 20.6 us, K = 30000 77.3 -> 44.8 us.
//
// With ucols != 0, ucols more CTAs per vector form u = e^T Q (64 columns
// each, the t rows over four row groups as in k_verify_u): u needs e alone,
// so it runs beside the scan instead of after the syndrome.
// -----------------------------------------------------------------------------
constexpr int kTileUCols = 64, kTileUGroups = kScanThreads / kTileUCols;
struct TileArgs {
    pvmvmd_key key;
    uint32_t tag, N, t, count;
    uint64_t idx0;
    const uint32_t *pi2inv, *v2p, *v1m;
    uint32_t *sparse_out, *F;
    unsigned long long *status;
    uint32_t *err;
    uint32_t skip_tile, spin_limit;
    const uint32_t *Qm;  // u = e^T Q where ucols != 0
    int K;
    uint32_t ucols;
    uint32_t *u;
};
// CTA `block` of count * (ntiles + ucols): the scan's first, then u's.
__device__ __forceinline__ void syndrome_tile(const TileArgs &A, uint32_t block) {
    const uint32_t N = A.N, t = A.t, ucols = A.ucols;
    const int K = A.K;
    __shared__ __align__(16) uint32_t s_list[kTileMaxT];
    __shared__ uint32_t s_val[kTileMaxT];
    // the keystream, then the sorted support and the suffix sums of the values
    __shared__ uint32_t s_words[2 * kTileMaxT + 1];
    static_assert(kTileMaxT == 512, "a draw's 512 words of keystream");
    uint32_t *s_supp = s_words, *s_suf = s_words + kTileMaxT;
    __shared__ uint32_t s_wsum[kScanThreads / 32], s_agg, s_prefix;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nw = kScanThreads / 32;
    const uint32_t ntiles = scan_tiles(N), nscan = A.count * ntiles;
    const bool scan = block < nscan;
    const uint32_t vec = scan ? block / ntiles : (block - nscan) / ucols;
    const uint32_t tile = scan ? ntiles - 1 - block % ntiles : 0u;  // from the end of the vector

    const uint32_t base = tile * kScanTile + tid * kScanItems;
    uint32_t idx[kScanItems], scale[kScanItems];
    if (scan) {
        if (base + kScanItems <= N) {
#pragma unroll
            for (int h = 0; h < kScanItems; h += 4) {
                const uint4 a = __ldg(reinterpret_cast<const uint4 *>(A.pi2inv + base + h));
                const uint4 b = __ldg(reinterpret_cast<const uint4 *>(A.v2p + base + h));
                idx[h] = a.x; idx[h + 1] = a.y; idx[h + 2] = a.z; idx[h + 3] = a.w;
                scale[h] = b.x; scale[h + 1] = b.y; scale[h + 2] = b.z; scale[h + 3] = b.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kScanItems; ++i) {
                const bool ok = base + i < N;
                idx[i] = ok ? __ldg(A.pi2inv + base + i) : 0u;
                scale[i] = ok ? __ldg(A.v2p + base + i) : 0u;
            }
        }
    }

    // ---- e: warp 0 the support, warp 1 the values
    const uint64_t vidx = A.idx0 + vec;
    if (warp == 0) warp_sample_support_short(A.key, A.tag, 2 * vidx, N, t, s_words, s_list, lane);
    else if (warp == 1) warp_sample_values(A.key, A.tag, 2 * vidx + 1, t, s_words + 512, s_val, lane);
    __syncthreads();
    if (warp == nw - 1) {  // s_suf[j] = sum_{j' >= j} e_{j'}; s_suf[t] = 0
        const uint32_t per = (t + 31) / 32;
        const uint32_t lo = min(t, lane * per), hi = min(t, lo + per);
        uint32_t sum = 0;
        for (uint32_t j = hi; j-- > lo;) sum = fadd(sum, s_val[j]);
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, incl, o);
            if (lane + o < 32) incl = fadd(incl, y);
        }
        uint32_t run = fsub(incl, sum);
        for (uint32_t j = hi; j-- > lo;) {
            run = fadd(run, s_val[j]);
            s_suf[j] = run;
        }
        if (lane == 0) s_suf[t] = 0;
    }
    for (uint32_t i = tid; i < t; i += kScanThreads) {  // ascending support by rank (entries distinct, unused slots larger)
        const uint32_t v = s_list[i];
        uint32_t rk = 0;
        for (uint32_t h = 0; h < t; h += 4) {
            const uint4 a = *reinterpret_cast<const uint4 *>(s_list + h);
            rk += (a.x < v) + (a.y < v) + (a.z < v) + (a.w < v);
        }
        s_supp[rk] = v;
    }
    __syncthreads();

    if (!scan) {
        // ---- u: 64 columns, the t rows over four groups
        __shared__ uint32_t s_part[kTileUGroups - 1][kTileUCols];
        const int grp = tid / kTileUCols, c = tid % kTileUCols;
        const int k = (int)((block - nscan) % ucols) * kTileUCols + c;
        const uint32_t per = (t + kTileUGroups - 1) / kTileUGroups;
        const uint32_t j0 = min(t, (uint32_t)grp * per), j1 = min(t, j0 + per);
        uint64_t acc = 0;
        if (k < K) {
            uint32_t j = j0;
            for (; j + 8 <= j1; j += 8) {
                uint32_t v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = __ldg(A.Qm + (size_t)s_supp[j + i] * K + k);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    acc += (uint64_t)s_val[j + i] * v[i];
                    if (i & 1) acc = fred(acc);
                }
            }
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = j + i < j1 ? __ldg(A.Qm + (size_t)s_supp[j + i] * K + k) : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (j + i < j1) acc += (uint64_t)s_val[j + i] * v[i];
                if (i & 1) acc = fred(acc);
            }
        }
        if (grp > 0) s_part[grp - 1][c] = (uint32_t)acc;
        __syncthreads();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (grp == 0 && k < K) {
            uint32_t sum = (uint32_t)acc;
#pragma unroll
            for (int g = 0; g < kTileUGroups - 1; ++g) sum = fadd(sum, s_part[g][c]);
            A.u[(size_t)vec * K + k] = sum;
        }
        return;
    }

    // ---- c over the tile, suffix sums inside it
    uint32_t c[kScanItems];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        uint32_t lo = 0, hi = t;  // first support index >= idx[i]
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_supp[mid] < idx[i]) lo = mid + 1; else hi = mid;
        }
        c[i] = fmul(scale[i], s_suf[lo]);  // 0 past N (scale 0)
    }
    uint32_t run = 0;
#pragma unroll
    for (int i = kScanItems - 1; i >= 0; --i) {
        run = fadd(run, c[i]);
        c[i] = run;
    }
    uint32_t w1[kScanItems];  // requested here, used after the look-back
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) w1[i] = base + i < N ? __ldg(A.v1m + base + i) : 0u;
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(kFull, incl, o);
        if (lane + o < 32) incl = fadd(incl, y);
    }
    if (lane == 0) s_wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t wv = lane < nw ? s_wsum[lane] : 0u;
        uint32_t winc = wv;
#pragma unroll
        for (int o = 1; o < nw; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, winc, o);
            if (lane + o < 32) winc = fadd(winc, y);
        }
        __syncwarp();
        if (lane < nw) s_wsum[lane] = fsub(winc, wv);
        if (lane == 0) s_agg = winc;
    }
    // everything so far came from the key and the tables; what the kernels
    // before this one may still use is written from here on
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    unsigned long long *st = A.status + (size_t)vec * ntiles;
    if (warp == 0) {
        // a failure-path test withholds one tile's word, so that the waits of
        // the tiles before it run out (off: skip_tile >= ntiles)
        if (lane == 0 && tile != A.skip_tile) st_relaxed_u64(st + tile, (1ull << 32) | s_agg);
        uint32_t sum = 0;
        for (uint32_t p = tile + 1 + lane; p < ntiles; p += 32) {
            uint32_t spins = 0;
            for (;;) {
                const unsigned long long w = ld_relaxed_u64(st + p);
                if (w >> 32) {
                    sum = fadd(sum, (uint32_t)w);
                    break;
                }
                if (++spins > A.spin_limit) {
                    record_error(A.err, kErrScanTimeout);
                    break;
                }
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sum = fadd(sum, __shfl_xor_sync(kFull, sum, o));
        if (lane == 0) s_prefix = sum;
    }
    if (A.sparse_out && tile == 0) {
        uint32_t *so = A.sparse_out + (size_t)vec * 2 * t;
        for (uint32_t j = tid; j < t; j += kScanThreads) {
            so[j] = s_supp[j];
            so[t + j] = s_val[j];
        }
    }
    __syncthreads();
    const uint32_t add = fadd(fadd(fsub(incl, run), s_wsum[warp]), s_prefix);
    uint32_t *Fv = A.F + (size_t)vec * N;
    uint32_t f[kScanItems];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) f[i] = fmul_mont(fadd(c[i], add), w1[i]);
    if (base + kScanItems <= N && N % 4 == 0) {
#pragma unroll
        for (int h = 0; h < kScanItems; h += 4)
            *reinterpret_cast<uint4 *>(Fv + base + h) = make_uint4(f[h], f[h + 1], f[h + 2], f[h + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < kScanItems; ++i)
            if (base + i < N) Fv[base + i] = f[i];
    }
}

}  // namespace
}  // namespace pv
