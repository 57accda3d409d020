// Client decode and verification (Protocol 3, Verify and Decrypt).
//
//  * k_decode           a large call in one kernel: the challenges, then the
//                       columns of k_decrypt and the checks.
//  * k_verify_u         u_q = e_q^T Q for the ell shared challenges
//                       (sum of t_y rows of Q, cost (2t-1)n per repetition,
//                       the e^T Q row of the cost table in Sec. 5.3).
//  * k_decrypt          Y_b = y_hat_b - P e_x,b (t_x rows of P^T), many
//                       short CTAs: 512, 256 or 64 columns of one vector
//                       each, the rows split over groups; in boost mode
//                       (Sec. 7.2) P e_x,b was prepared ahead and is read
//                       instead of the t_x rows of P^T.
//  * k_check            accept_b = AND_q (L_q == R_q), L_q = u_q . x_hat_b,
//                       R_q = g_q . y_hat_b with g_q = G_y e_q, so that
//                       R_q = e_q^T (G_y^T y_hat_b) by transposition.
//  * k_output_mask      the output masks P e_x,b alone (boost mode's
//                       offline step).
#include <cmath>
#include <map>
#include <mutex>

#include <cooperative_groups.h>

#include "common.cuh"
#include "launch.h"
#include "syndrome.cuh"

namespace cg = cooperative_groups;

namespace pv {
namespace {

constexpr int kDecThreads = 256;

// A row of P^T is read once by a CTA, so L1 would only be filled in vain
// (decode of 4096 x 4096, 100 vectors: 45.1 -> 41.2 us without; asking L2 for
// 256 bytes at a time 43.0).
__device__ __forceinline__ uint4 ldg4(const uint32_t *p) {
    uint4 v;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}

// u[q][k] = sum_j chal_val[q][j] Q[chal_supp[q][j]][k]: a CTA covers 64
// columns with the t rows split over four row groups (so a thread streams
// about t/4 rows, one round of loads for t = 31), the groups' sums meeting
// in shared memory.
constexpr int kVuCols = 64, kVuGroups = 4;
__global__ void __launch_bounds__(kVuCols * kVuGroups) k_verify_u(const uint32_t *__restrict__ Qm, int K,
                                                                 const uint32_t *chal, uint32_t t, uint32_t *u) {
    extern __shared__ uint32_t sm[];
    __shared__ uint32_t s_part[kVuGroups - 1][kVuCols];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the challenges come from the kernel before
    const uint32_t q = blockIdx.y;
    const int tid = threadIdx.x, grp = tid / kVuCols, c = tid % kVuCols;
    const uint32_t *ch = chal + (size_t)q * 2 * t;
    for (uint32_t j = tid; j < 2 * t; j += kVuCols * kVuGroups) sm[j] = ch[j];
    __syncthreads();
    const int k = blockIdx.x * kVuCols + c;
    const uint32_t per = (t + kVuGroups - 1) / kVuGroups;
    const uint32_t j0 = min(t, (uint32_t)grp * per), j1 = min(t, j0 + per);
    uint64_t acc = 0;
    if (k < K) {
        uint32_t j = j0;
        for (; j + 8 <= j1; j += 8) {
            uint32_t v[8];
#pragma unroll
            for (int s2 = 0; s2 < 8; ++s2) v[s2] = __ldg(Qm + (size_t)sm[j + s2] * K + k);
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) acc += (uint64_t)sm[t + j + s2] * v[s2];
            acc = fred(acc);
#pragma unroll
            for (int s2 = 4; s2 < 8; ++s2) acc += (uint64_t)sm[t + j + s2] * v[s2];
            acc = fred(acc);
        }
        for (; j < j1; ++j) acc = fred(acc + (uint64_t)sm[t + j] * __ldg(Qm + (size_t)sm[j] * K + k));
    }
    if (grp > 0) s_part[grp - 1][c] = (uint32_t)acc;
    __syncthreads();
    if (grp == 0 && k < K) {
        uint32_t sum = (uint32_t)acc;
#pragma unroll
        for (int g2 = 0; g2 < kVuGroups - 1; ++g2) sum = fadd(sum, s_part[g2][c]);
        u[(size_t)q * K + k] = sum;
    }
}

__device__ __forceinline__ uint32_t warp_fsum(uint32_t v) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = fadd(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// pe[s] = sum_j vals[j] P^T[supp[j]][i + s] mod q for the four columns
// i .. i+3 (columns at or past c1 read as 0); 16-byte loads when vec.
__device__ __forceinline__ void pe_cols(const uint32_t *__restrict__ PT, int m, const uint32_t *supp,
                                    const uint32_t *vals, uint32_t t_x, int i, int c1, bool vec,
                                    uint32_t pe[4]) {
    uint64_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    uint32_t j = 0;
    for (; j + 8 <= t_x; j += 8) {
        uint4 v[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const uint32_t *row = PT + (size_t)supp[j + s] * m + i;
            if (vec) {
                v[s] = ldg4(row);
            } else {
                v[s].x = row[0];
                v[s].y = i + 1 < c1 ? row[1] : 0u;
                v[s].z = i + 2 < c1 ? row[2] : 0u;
                v[s].w = i + 3 < c1 ? row[3] : 0u;
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int s = 4 * h; s < 4 * h + 4; ++s) {
                const uint64_t e = vals[j + s];
                a0 += e * v[s].x; a1 += e * v[s].y; a2 += e * v[s].z; a3 += e * v[s].w;
            }
            a0 = fred(a0); a1 = fred(a1); a2 = fred(a2); a3 = fred(a3);
        }
    }
    for (; j + 4 <= t_x; j += 4) {
        uint4 v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const uint32_t *row = PT + (size_t)supp[j + s] * m + i;
            if (vec) {
                v[s] = ldg4(row);
            } else {
                v[s].x = row[0];
                v[s].y = i + 1 < c1 ? row[1] : 0u;
                v[s].z = i + 2 < c1 ? row[2] : 0u;
                v[s].w = i + 3 < c1 ? row[3] : 0u;
            }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const uint64_t e = vals[j + s];
            a0 += e * v[s].x; a1 += e * v[s].y; a2 += e * v[s].z; a3 += e * v[s].w;
        }
        a0 = fred(a0); a1 = fred(a1); a2 = fred(a2); a3 = fred(a3);
    }
    for (; j < t_x; ++j) {
        const uint32_t *row = PT + (size_t)supp[j] * m + i;
        const uint64_t e = vals[j];
        a0 += e * row[0];
        if (i + 1 < c1) a1 += e * row[1];
        if (i + 2 < c1) a2 += e * row[2];
        if (i + 3 < c1) a3 += e * row[3];
    }
    pe[0] = fred(a0);
    pe[1] = fred(a1);
    pe[2] = fred(a2);
    pe[3] = fred(a3);
}

// ---------------------------------------------------------------------------
// Decrypt: Y_b = y_hat_b - P e_x,b.  A CTA owns 512 columns of one vector
// (128 column threads x 4 columns, so each row of P^T is read in 2 KiB
// segments) and splits the t_x rows over kDecGroups = 2 row groups, so each
// thread streams about t_x / 2 row segments (rounds of 8 loads in flight)
// and the grid holds many short CTAs whatever m and B are; or 256 columns
// over 4 row groups when that fills the last wave of resident CTAs better;
// or 64 columns over 16 when the whole grid is resident at once.  The groups'
// partial sums meet in shared memory.  (256 columns everywhere, or 1024
// columns and 1 group, were 6 and 13 % slower at m = K = 8192, B = 256.)
// In boost mode (Sec. 7.2) P e_x,b was prepared ahead: Y_b = y_hat_b - mask_b.
// The grid runs vectors fastest (blockIdx.x = b, blockIdx.y = column block),
// so the CTAs in flight share a few column blocks and a row of P^T drawn by
// several vectors' supports is read from HBM once and then from L2.
// ---------------------------------------------------------------------------
template <bool kBoost, int kDecGroups>
__device__ __forceinline__ void decrypt_cta(const uint32_t *__restrict__ PT, int m, const uint32_t *__restrict__ st,
                                            uint32_t t_x, uint32_t Nx, const uint32_t *Yhat, uint32_t *Y,
                                            const uint32_t *__restrict__ mask, bool vec, size_t b, uint32_t yblk) {
    constexpr int kDecColThreads = kDecThreads / kDecGroups;
    constexpr int kDecCols = 4 * kDecColThreads;
    extern __shared__ uint32_t sm[];  // support[t_x], values[t_x]
    __shared__ uint4 s_part[kDecGroups > 1 ? kDecGroups - 1 : 1][kDecColThreads];
    const int tid = threadIdx.x;
    const int grp = tid / kDecColThreads, ct = tid % kDecColThreads;
    // boost mode: no rows to split, every thread owns 4 of 1024 columns
    const int i = kBoost ? ((int)yblk * kDecThreads + tid) * 4 : (int)yblk * kDecCols + ct * 4;
    uint32_t pe[4] = {0u, 0u, 0u, 0u};
    if (!kBoost) {
        const uint32_t *stb = st + b * 2 * t_x;
        // a support index past the code (a state the encode did not write)
        // reads row 0 instead: the result is then wrong, never out of bounds
        for (uint32_t j = tid; j < 2 * t_x; j += kDecThreads) {
            const uint32_t v = stb[j];
            sm[j] = (j < t_x && v >= Nx) ? 0u : v;
        }
        __syncthreads();
        const uint32_t per = (t_x + kDecGroups - 1) / kDecGroups;
        const uint32_t j0 = min(t_x, (uint32_t)grp * per), j1 = min(t_x, j0 + per);
        if (i < m && j0 < j1) pe_cols(PT, m, sm + j0, sm + t_x + j0, j1 - j0, i, m, vec, pe);
        if (grp > 0) s_part[grp - 1][ct] = make_uint4(pe[0], pe[1], pe[2], pe[3]);
        __syncthreads();
        if (grp > 0) return;
#pragma unroll
        for (int g2 = 0; g2 < kDecGroups - 1; ++g2) {
            const uint4 v = s_part[g2][ct];
            pe[0] = fadd(pe[0], v.x);
            pe[1] = fadd(pe[1], v.y);
            pe[2] = fadd(pe[2], v.z);
            pe[3] = fadd(pe[3], v.w);
        }
    }
    if (i >= m) return;
    const uint32_t *yh = Yhat + b * m;
    uint32_t *yo = Y + b * m;
    if (kBoost) {
        const uint32_t *mk = mask + b * m;
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) pe[q2] = i + q2 < m ? mk[i + q2] : 0u;
    }
    if (vec) {
        // y_hat is read here rather than prefetched before the row loop: a
        // live uint4 across the loop raises the kernel to 70 registers and
        // four CTAs per SM to three
        const uint4 yv = *reinterpret_cast<const uint4 *>(yh + i);
        *reinterpret_cast<uint4 *>(yo + i) =
            make_uint4(fsub(yv.x, pe[0]), fsub(yv.y, pe[1]), fsub(yv.z, pe[2]), fsub(yv.w, pe[3]));
    } else {
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2)
            if (i + q2 < m) yo[i + q2] = fsub(yh[i + q2], pe[q2]);
    }
}

template <bool kBoost, int kDecGroups>
__global__ void __launch_bounds__(kDecThreads) k_decrypt(const uint32_t *__restrict__ PT, int m,
                                                        const uint32_t *__restrict__ st, uint32_t t_x,
                                                        uint32_t Nx, const uint32_t *Yhat, uint32_t *Y,
                                                        const uint32_t *__restrict__ mask, bool vec) {
    decrypt_cta<kBoost, kDecGroups>(PT, m, st, t_x, Nx, Yhat, Y, mask, vec, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Verify: accept_b = AND_q [ L_q == R_q ] with L_q = u_q . x_hat_b and
// R_q = g_q . y_hat_b (= e_q^T (G_y^T y_hat_b) by transposition), u_q =
// e_q^T Q and g_q = G_y e_q from the challenge kernels.  One cluster of up to
// eight CTAs per vector; the repetitions run one after the other over the (cached) vectors.
// ---------------------------------------------------------------------------
// The S CTAs of a cluster (256 threads, four loads of each operand in flight
// per thread) take one slice of the columns each and add their sums through
// distributed shared memory: small CTAs find room beside a decrypt's (one CTA
// of 512 threads per vector took 15.5 us cold for 14336 x 4096, 64 vectors).
constexpr int kCheckThreads = 256;
constexpr int kCheckBatch = 4;      // loads in flight per operand and thread
constexpr int kCheckSlice = 2048;   // columns a CTA takes, where eight CTAs suffice
constexpr int kCheckMaxCluster = 8;

__global__ void __launch_bounds__(kCheckThreads, 4) k_check(const uint32_t *Xhat, int K, const uint32_t *Yhat,
                                                           int m, const uint32_t *g, const uint32_t *u, uint32_t ell,
                                                           int32_t *accept) {
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ uint32_t s_part[4][kCheckThreads / 32];
    __shared__ uint32_t s_sum[4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t S = cluster.num_blocks(), rank = cluster.block_rank();
    const size_t b = blockIdx.y;
    const uint32_t *xh = Xhat + b * K, *yh = Yhat + b * m;
    // the kernel after this one (the next call's encode) may start its
    // key-only work now; g and u come from the kernels before
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = K > m ? K : m;
    const int per = (n + (int)S - 1) / (int)S;
    const int n0 = (int)rank * per, n1 = min(n, n0 + per);
    int ok = 1;
    // two repetitions per pass: x_hat and y_hat are read once per pair
    for (uint32_t q = 0; q < ell; q += 2) {
        const bool two = q + 1 < ell;
        const uint32_t *u0 = u + (size_t)q * K, *g0 = g + (size_t)q * m;
        const uint32_t *u1 = two ? u0 + K : u0, *g1 = two ? g0 + m : g0;
        uint64_t l0 = 0, l1 = 0, r0 = 0, r1 = 0;
        for (int k0 = n0 + tid; k0 < n1; k0 += kCheckBatch * kCheckThreads) {
            uint32_t x[kCheckBatch], y[kCheckBatch], a0[kCheckBatch], a1[kCheckBatch], c0[kCheckBatch],
                c1[kCheckBatch];
#pragma unroll
            for (int v = 0; v < kCheckBatch; ++v) {
                const int k = k0 + v * kCheckThreads;
                const bool kx = k < n1 && k < K, ky = k < n1 && k < m;
                x[v] = kx ? xh[k] : 0u;
                a0[v] = kx ? __ldcg(u0 + k) : 0u;
                a1[v] = kx ? __ldcg(u1 + k) : 0u;
                y[v] = ky ? yh[k] : 0u;
                c0[v] = ky ? __ldcg(g0 + k) : 0u;
                c1[v] = ky ? __ldcg(g1 + k) : 0u;
            }
            // four products of values below q stay below 2^64 with the
            // reduced running sum
            static_assert(kCheckBatch <= 4, "sums reduced after at most four products");
#pragma unroll
            for (int v = 0; v < kCheckBatch; ++v) {
                l0 += (uint64_t)a0[v] * x[v];
                l1 += (uint64_t)a1[v] * x[v];
                r0 += (uint64_t)c0[v] * y[v];
                r1 += (uint64_t)c1[v] * y[v];
            }
            l0 = fred(l0);
            l1 = fred(l1);
            r0 = fred(r0);
            r1 = fred(r1);
        }
        const uint32_t w0 = warp_fsum((uint32_t)l0), w1 = warp_fsum((uint32_t)l1);
        const uint32_t w2 = warp_fsum((uint32_t)r0), w3 = warp_fsum((uint32_t)r1);
        if (lane == 0) {
            s_part[0][warp] = w0;
            s_part[1][warp] = w1;
            s_part[2][warp] = w2;
            s_part[3][warp] = w3;
        }
        __syncthreads();
        if (tid < 4) {
            uint32_t sum = 0;
            for (int w = 0; w < kCheckThreads / 32; ++w) sum = fadd(sum, s_part[tid][w]);
            s_sum[tid] = sum;
        }
        cluster.sync();
        if (rank == 0 && tid == 0) {
            uint32_t t[4] = {0u, 0u, 0u, 0u};
            for (uint32_t c = 0; c < S; ++c) {
                const uint32_t *ps = cluster.map_shared_rank(s_sum, c);
#pragma unroll
                for (int i = 0; i < 4; ++i) t[i] = fadd(t[i], ps[i]);
            }
            ok &= (t[0] == t[2]);
            if (two) ok &= (t[1] == t[3]);
        }
        cluster.sync();  // the sums are read before a CTA writes the next ones or exits
    }
    if (rank == 0 && tid == 0) accept[b] = ok;
}

// ---------------------------------------------------------------------------
// A large decode in one kernel: CTAs of 256 threads, by index
//   the challenges' tiles and u = e^T Q (syndrome_tile),
//   g = G_y e from the finished tiles,
//   the decrypt, all but its last wave of resident CTAs,
//   the check of one vector each, from u and g,
//   the rest of the decrypt.
// A CTA waits only for CTAs of lower index (started first, as in
// syndrome_tile); the verification is done while P^T streams, and nothing is
// left between two decodes but one launch (a side stream for the verification,
// forked and joined by events, kept them 6 to 10 us apart).  sync: the finished
// tiles of each challenge, the finished CTAs of u and g, the CTAs of the
// verification that are through; all zero at launch, and set back, with the
// tiles' status words, by the last of those.  A wait that runs out lets its CTA
// go on, so only a count of all of them says that none will use the words again
// (4096 x 4096, 100 vectors 41.6 -> 41.8 us against a count of the checks).
// ---------------------------------------------------------------------------
constexpr int kSyncReady = 16, kSyncFinished = 17;
static_assert(kSyncFinished < kDecodeSyncWords, "sync words");

struct DecodeArgs {
    TileArgs tile;
    const uint32_t *pi1inv;
    uint32_t r, B, tiles, gather, first, decrypt;  // CTAs of each part; `first` of the decrypt's before the checks
    uint32_t *g;
    const uint32_t *PT, *st, *Xhat, *Yhat;
    uint32_t *Y;
    int m;
    uint32_t t_x, Nx;
    int32_t *accept;
    uint32_t *sync;
    bool vec;
};

// The CTA's writes before this are visible to a CTA whose sync_await sees it.
__device__ __forceinline__ void sync_signal(uint32_t *p) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(p, 1u);
    }
}
__device__ __forceinline__ void sync_await(const uint32_t *p, uint32_t n, uint32_t *err, uint32_t spin_limit) {
    if (threadIdx.x == 0) {
        uint32_t spins = 0;
        while (ld_acquire_u32(p) < n) {
            if (++spins > spin_limit) {
                record_error(err, kErrScanTimeout);
                break;
            }
            __nanosleep(64);
        }
    }
    __syncthreads();
}
// The last thing that a CTA of the verification does with sync and the status
// words; the last of them sets both back.  The fence orders a signal before it;
// a check signals nothing and has read what it waits for.
__device__ __forceinline__ void sync_leave(const DecodeArgs &a, uint32_t nscan, bool signalled) {
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        if (signalled) __threadfence();
        s_last = atomicAdd(a.sync + kSyncFinished, 1u) == a.tiles + a.gather + a.B - 1;
        if (s_last) __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    for (uint32_t i = threadIdx.x; i < nscan; i += kDecThreads) a.tile.status[i] = 0ull;
    if (threadIdx.x < kDecodeSyncWords) a.sync[threadIdx.x] = 0u;
}

// accept_b, by one CTA (as k_check with a cluster of one)
__device__ __forceinline__ void check_cta(const DecodeArgs &a, uint32_t b) {
    __shared__ uint32_t s_part[4][kDecThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = a.tile.K, m = a.m, n = K > m ? K : m;
    const uint32_t *xh = a.Xhat + (size_t)b * K, *yh = a.Yhat + (size_t)b * m;
    int ok = 1;
    for (uint32_t q = 0; q < a.tile.count; q += 2) {
        const bool two = q + 1 < a.tile.count;
        const uint32_t *u0 = a.tile.u + (size_t)q * K, *g0 = a.g + (size_t)q * m;
        const uint32_t *u1 = two ? u0 + K : u0, *g1 = two ? g0 + m : g0;
        uint64_t l0 = 0, l1 = 0, r0 = 0, r1 = 0;
        for (int k0 = tid; k0 < n; k0 += 4 * kDecThreads) {
            uint32_t x[4], y[4], a0[4], a1[4], c0[4], c1[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int k = k0 + v * kDecThreads;
                const bool kx = k < K, ky = k < m;
                x[v] = kx ? xh[k] : 0u;
                a0[v] = kx ? __ldcg(u0 + k) : 0u;
                a1[v] = kx ? __ldcg(u1 + k) : 0u;
                y[v] = ky ? yh[k] : 0u;
                c0[v] = ky ? __ldcg(g0 + k) : 0u;
                c1[v] = ky ? __ldcg(g1 + k) : 0u;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {  // four products and the reduced sum stay below 2^64
                l0 += (uint64_t)a0[v] * x[v];
                l1 += (uint64_t)a1[v] * x[v];
                r0 += (uint64_t)c0[v] * y[v];
                r1 += (uint64_t)c1[v] * y[v];
            }
            l0 = fred(l0);
            l1 = fred(l1);
            r0 = fred(r0);
            r1 = fred(r1);
        }
        const uint32_t w[4] = {warp_fsum((uint32_t)l0), warp_fsum((uint32_t)l1), warp_fsum((uint32_t)r0),
                               warp_fsum((uint32_t)r1)};
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i) s_part[i][warp] = w[i];
        __syncthreads();
        if (tid == 0) {
            uint32_t t[4] = {0u, 0u, 0u, 0u};
            for (int i = 0; i < 4; ++i)
                for (int v = 0; v < kDecThreads / 32; ++v) t[i] = fadd(t[i], s_part[i][v]);
            ok &= (t[0] == t[2]);
            if (two) ok &= (t[1] == t[3]);
        }
        __syncthreads();
    }
    if (tid == 0) a.accept[b] = ok;
}

template <int kDecGroups>
__global__ void __launch_bounds__(kDecThreads, 4) k_decode(const __grid_constant__ DecodeArgs a) {
    static_assert(kDecThreads == kScanThreads, "one block size for every part");
    uint32_t blk = blockIdx.x;
    const uint32_t ntiles = scan_tiles(a.tile.N), nscan = a.tile.count * ntiles;
    if (blk < a.tiles) {
        syndrome_tile(a.tile, blk);
        // a failure-path test withholds one tile's signal too (off: skip_tile >= ntiles)
        if (blk >= nscan || ntiles - 1 - blk % ntiles != a.tile.skip_tile)
            sync_signal(a.sync + (blk < nscan ? blk / ntiles : (uint32_t)kSyncReady));
        else
            __syncthreads();
        sync_leave(a, nscan, true);
        return;
    }
    blk -= a.tiles;
    if (blk < a.gather) {
        const uint32_t per = a.gather / a.tile.count, q = blk / per, j = blk % per * kDecThreads + threadIdx.x;
        const uint32_t *p = a.pi1inv + (size_t)j * a.r;
        uint32_t at[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (a.r == 8 && j < (uint32_t)a.m) {
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(p)), y = __ldg(reinterpret_cast<const uint4 *>(p + 4));
            at[0] = x.x; at[1] = x.y; at[2] = x.z; at[3] = x.w;
            at[4] = y.x; at[5] = y.y; at[6] = y.z; at[7] = y.w;
        }
        sync_await(a.sync + q, ntiles, a.tile.err, a.tile.spin_limit);
        if (j < (uint32_t)a.m) {
            const uint32_t *F = a.tile.F + (size_t)q * a.tile.N;
            uint32_t s = 0;
            if (a.r == 8) {
                uint32_t f[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) f[c] = __ldcg(F + at[c]);
#pragma unroll
                for (int c = 0; c < 8; ++c) s = fadd(s, f[c]);
            } else {
                for (uint32_t c = 0; c < a.r; ++c) s = fadd(s, __ldcg(F + __ldg(p + c)));
            }
            a.g[(size_t)q * a.m + j] = s;
        }
        sync_signal(a.sync + kSyncReady);
        sync_leave(a, nscan, true);
        return;
    }
    blk -= a.gather;
    if (blk >= a.first && blk < a.first + a.B) {
        sync_await(a.sync + kSyncReady, a.tiles - nscan + a.gather, a.tile.err, a.tile.spin_limit);
        check_cta(a, blk - a.first);
        sync_leave(a, nscan, false);
        return;
    }
    if (blk >= a.first) blk -= a.B;
    decrypt_cta<false, kDecGroups>(a.PT, a.m, a.st, a.t_x, a.Nx, a.Yhat, a.Y, nullptr, a.vec, blk % a.B, blk / a.B);
}

// out[b][col] = (P e_x,b)_col for the columns of this CTA (1024 per CTA).
__global__ void __launch_bounds__(kDecThreads) k_output_mask(const uint32_t *__restrict__ PT, int m,
                                                            const uint32_t *__restrict__ st, uint32_t t_x,
                                                            uint32_t *__restrict__ out, bool vec) {
    extern __shared__ uint32_t sm[];  // support[t_x], values[t_x]
    const size_t b = blockIdx.y;
    const uint32_t *stb = st + b * 2 * t_x;
    for (uint32_t j = threadIdx.x; j < 2 * t_x; j += kDecThreads) sm[j] = stb[j];
    __syncthreads();
    const int i = (int)blockIdx.x * kDecThreads * 4 + (int)threadIdx.x * 4;
    if (i >= m) return;
    uint32_t pe[4];
    pe_cols(PT, m, sm, sm + t_x, t_x, i, m, vec, pe);
#pragma unroll
    for (int s = 0; s < 4; ++s)
        if (i + s < m) out[b * m + i + s] = pe[s];
}

// out = a + b over F_q, n elements, 16 bytes per thread where aligned.
__global__ void __launch_bounds__(256) k_field_add(const uint32_t *a, const uint32_t *b, size_t n,
                                                  uint32_t *out, bool vec) {
    const size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) * 4;
    if (i >= n) return;
    if (vec && i + 4 <= n) {
        const uint4 x = *reinterpret_cast<const uint4 *>(a + i);
        const uint4 y = *reinterpret_cast<const uint4 *>(b + i);
        *reinterpret_cast<uint4 *>(out + i) = make_uint4(fadd(x.x, y.x), fadd(x.y, y.y), fadd(x.z, y.z), fadd(x.w, y.w));
    } else {
        for (size_t k = i; k < n && k < i + 4; ++k) out[k] = fadd(a[k], b[k]);
    }
}

}  // namespace

cudaError_t launch_field_add(const uint32_t *a, const uint32_t *b, size_t n, uint32_t *out,
                             cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const bool vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) |
                       reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
    const size_t blocks = (n + 1023) / 1024;
    if (blocks > 0x7fffffffu) return cudaErrorInvalidValue;
    k_field_add<<<(unsigned)blocks, 256, 0, s>>>(a, b, n, out, vec); note_launch();
    return cudaGetLastError();
}

cudaError_t launch_output_mask(const uint32_t *PT, int m, const uint32_t *st, uint32_t t_x, int B,
                               uint32_t *out, cudaStream_t s) {
    if (B <= 0 || m <= 0) return cudaSuccess;
    const bool vec = (m % 4 == 0) && ((reinterpret_cast<uintptr_t>(PT) & 15u) == 0);
    for (int b0 = 0; b0 < B; b0 += 65535) {
        const int nb = B - b0 < 65535 ? B - b0 : 65535;
        dim3 grid((m + kDecThreads * 4 - 1) / (kDecThreads * 4), nb);
        k_output_mask<<<grid, kDecThreads, 2 * (size_t)t_x * sizeof(uint32_t), s>>>(
            PT, m, st + (size_t)b0 * 2 * t_x, t_x, out + (size_t)b0 * m, vec); note_launch();
    }
    return cudaGetLastError();
}

cudaError_t launch_verify_u(const uint32_t *Qm, int K, const uint32_t *chal, uint32_t t_y,
                            uint32_t ell, uint32_t *u, cudaStream_t s) {
    if (K <= 0 || ell == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((K + kVuCols - 1) / kVuCols, ell, 1);
    cfg.blockDim = dim3(kVuCols * kVuGroups, 1, 1);
    cfg.dynamicSmemBytes = 2 * (size_t)t_y * sizeof(uint32_t);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return counted_launch(cudaLaunchKernelEx(&cfg, k_verify_u, Qm, K, chal, t_y, u));
}

// Resident k_decrypt CTAs on the current device (cached per device).
int decrypt_slots() {
    static std::mutex mu;
    static std::map<int, int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(dev);
    if (it != cache.end()) return it->second;
    int per_sm = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_decrypt<false, 2>, kDecThreads, 1024) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        per_sm = 0;
    }
    return cache[dev] = per_sm * sms;
}

// Columns per CTA of a decrypt.
int decrypt_cols(int m, int B) {
    // Every CTA streams the same t_x row segments, so a last wave that is a
    // third full costs as much as a full one: 256-column CTAs are used when
    // they fill the last wave of resident CTAs clearly better than 512
    // (4096 x 4096, 100 vectors: 800 CTAs are 1.32 waves of 608, 1600 are
    // 2.63; decrypt 47 -> 41 us, step 0.3221 -> 0.3202 ms).  Where both
    // fill alike the wider CTAs stay (70B-class shapes, 256 vectors: 256
    // columns everywhere took 2.221 -> 2.272 ms per step).
    // Where 64-column CTAs, with the rows over 16 groups, fit the GPU at once
    // they are used: a thread then waits for about t_x / 128 rounds of eight
    // rows instead of t_x / 16 (256 x 256, one vector: 15.7 -> 5 us cold).
    const int slots = decrypt_slots();
    auto fill = [&](int cols) {
        const double waves = (double)B * (double)((m + cols - 1) / cols) / slots;
        return waves / std::ceil(waves);
    };
    const bool once = slots > 0 && (double)B * (double)((m + 63) / 64) <= slots;
    return once ? 64 : slots > 0 && fill(256) > fill(512) + 0.1 ? 256 : 512;
}

cudaError_t launch_decode(const DecodeCall &c, cudaStream_t s) {
    const int cols = decrypt_cols(c.m, c.B);
    const uint32_t ntiles = scan_tiles(c.Ny), ucols = (uint32_t)(c.K + kTileUCols - 1) / kTileUCols;
    const uint64_t dec = (uint64_t)c.B * ((c.m + cols - 1) / cols);
    const uint64_t tiles = (uint64_t)c.ell * (ntiles + ucols), gather = (uint64_t)c.ell * ((c.m + 255) / 256);
    if (tiles + gather + dec + c.B > 0x7fffffffu) return cudaErrorInvalidValue;
    const size_t smem = 2 * (size_t)c.t_x * sizeof(uint32_t);
    if (smem > 32 * 1024) return cudaErrorInvalidValue;
    const DebugWait dbg = debug_wait();
    const bool inject = dbg.site == PVMVMD_DEBUG_WAIT_SCAN;
    DecodeArgs a{};
    a.tile = TileArgs{c.key, c.tag, c.Ny, c.t_y, c.ell, 0, c.pi2inv, c.v2p, c.v1m, nullptr, c.F, c.status, c.err,
                      inject ? dbg.index : 0xFFFFFFFFu, inject ? (uint32_t)dbg.limit : kSpinLimit, c.Q, c.K, ucols, c.u};
    a.pi1inv = c.pi1inv;
    a.r = c.r;
    a.B = (uint32_t)c.B;
    a.tiles = (uint32_t)tiles;
    a.gather = (uint32_t)gather;
    a.decrypt = (uint32_t)dec;
    a.first = dec > (uint64_t)decrypt_slots() ? (uint32_t)(dec - decrypt_slots()) : 0u;
    a.g = c.g;
    a.PT = c.PT;
    a.st = c.st;
    a.Xhat = c.Xhat;
    a.Yhat = c.Yhat;
    a.Y = c.Y;
    a.m = c.m;
    a.t_x = c.t_x;
    a.Nx = c.Nx;
    a.accept = c.accept;
    a.sync = c.sync;
    a.vec = c.m % 4 == 0 && ((reinterpret_cast<uintptr_t>(c.PT) | reinterpret_cast<uintptr_t>(c.Yhat) |
                              reinterpret_cast<uintptr_t>(c.Y)) & 15u) == 0;
    const auto kern = cols == 256 ? k_decode<4> : k_decode<2>;
    kern<<<a.tiles + a.gather + a.decrypt + a.B, kDecThreads, smem, s>>>(a); note_launch();
    return cudaGetLastError();
}

bool decode_wins(int m, int B, uint32_t t_x, uint32_t t_y, uint32_t ell) {
    // a decrypt of more than one wave of resident CTAs
    const int cols = decrypt_cols(m, B), slots = decrypt_slots();
    return slots > 0 && cols > 64 && syndrome_tiles_eligible(t_y) && ell <= 16 && 2 * t_x * 4 <= 32 * 1024 &&
           (uint64_t)B * ((m + cols - 1) / cols) > (uint64_t)slots;
}

cudaError_t launch_decrypt(const uint32_t *PT, int m, const uint32_t *st, uint32_t t_x, uint32_t Nx,
                           const uint32_t *Yhat, int B, uint32_t *Y, cudaStream_t s, const uint32_t *mask) {
    if (B <= 0 || m <= 0) return cudaSuccess;
    const bool vec = (m % 4 == 0) &&
                     ((reinterpret_cast<uintptr_t>(PT) | reinterpret_cast<uintptr_t>(Yhat) |
                       reinterpret_cast<uintptr_t>(Y)) & 15u) == 0;
    const size_t smem = mask ? 0 : 2 * (size_t)t_x * sizeof(uint32_t);
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    const dim3 grid_mask((unsigned)B, (m + 4 * kDecThreads - 1) / (4 * kDecThreads));
    if (mask) {
        k_decrypt<true, 2><<<grid_mask, kDecThreads, 0, s>>>(PT, m, nullptr, t_x, Nx, Yhat, Y, mask, vec);
        note_launch();
        return cudaGetLastError();
    }
    const int cols = decrypt_cols(m, B);
    if ((m + cols - 1) / cols > 65535) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)B, (m + cols - 1) / cols);
    if (cols == 64)
        k_decrypt<false, 16><<<grid, kDecThreads, smem, s>>>(PT, m, st, t_x, Nx, Yhat, Y, nullptr, vec);
    else if (cols == 256)
        k_decrypt<false, 4><<<grid, kDecThreads, smem, s>>>(PT, m, st, t_x, Nx, Yhat, Y, nullptr, vec);
    else
        k_decrypt<false, 2><<<grid, kDecThreads, smem, s>>>(PT, m, st, t_x, Nx, Yhat, Y, nullptr, vec);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_check(const uint32_t *Xhat, int K, const uint32_t *Yhat, int m, const uint32_t *g,
                         const uint32_t *u, uint32_t ell, int B, int32_t *accept, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    const int n = K > m ? K : m;
    unsigned S = 1;
    while (S < (unsigned)kCheckMaxCluster && (int64_t)S * kCheckSlice < n) S *= 2;
    for (int b0 = 0; b0 < B; b0 += 65535) {
        const int nb = B - b0 < 65535 ? B - b0 : 65535;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(S, (unsigned)nb, 1);
        cfg.blockDim = dim3(kCheckThreads, 1, 1);
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = S;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        const cudaError_t e = counted_launch(cudaLaunchKernelEx(&cfg, k_check, Xhat + (size_t)b0 * K, K,
                                                                Yhat + (size_t)b0 * m, m, g, u, ell, accept + b0));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace pv
