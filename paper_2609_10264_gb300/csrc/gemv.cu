// Batch-1 field GEMV: y_hat = M x_hat over F_q (the server's online work,
// Sec. 6.1), M int8 m x K row-major, x_hat canonical uint32.
//
// One byte of M per field MAC, so HBM bounds it.  x_hat centred is split into
// four signed base-256 digits (d0 + 2^8 d1 + 2^16 d2 + 2^24 d3), so a field
// MAC becomes four int8 x int8 products done by dp4a, four columns per
// instruction, with exact int32 sums (|sum| <= 128*128*K < 2^31), combined in
// int64 and reduced mod q once per row.
//  * k_gemv_ring   K a multiple of 16 and 16-byte aligned rows: a list of
//                  independent products in one launch.
//  * k_gemv        any K and alignment, words and funnel shifts, one product.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "launch.h"

namespace pv {
namespace {

constexpr int kGemvThreads = 512;
// Digit planes of a K segment live in shared memory (4 bytes per column); a
// longer K is done in segments whose mod-q partial results are added.
constexpr int kGemvMaxK = 48 * 1024;

// Sum of v[index] over the 32 lanes, where index = lane / (32 / V): after the
// call every lane holds the total of the entry its lane number selects.
template <int V>
__device__ __forceinline__ int transposed_reduce(int (&v)[V], int lane) {
#pragma unroll
    for (int n = V, o = 16; n > 1; n >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const int send = upper ? v[i] : v[i + n / 2];
            const int keep = upper ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, send, o);
        }
    }
    int x = v[0];
#pragma unroll
    for (int o = 16 / V; o >= 1; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

template <int ROWS, int UNROLL>
__global__ void __launch_bounds__(kGemvThreads, 1)
    k_gemv(const int8_t *__restrict__ W, size_t ldw, int m, int K, const uint32_t *__restrict__ xhat,
           uint32_t *__restrict__ y, bool accumulate) {
    extern __shared__ uint4 s_planes[];  // 4 planes of nchunks 16-byte chunks
    const int nchunks = (K + 15) / 16;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nwarps = kGemvThreads / 32;
    constexpr int V = ROWS * 4;
    static_assert(V <= 32 && (V & (V - 1)) == 0, "ROWS must be 1, 2, 4 or 8");

    const int ngroups = (m + ROWS - 1) / ROWS;
    const int gstride = gridDim.x * nwarps;
    int g = warp * gridDim.x + blockIdx.x;

    // Issue the first batch of M loads before building the digit planes (bytes
    // past K meet zero digits).
    const int8_t *W_end = W + (size_t)(m - 1) * ldw + K;
    uint4 wbuf[UNROLL][ROWS];
    auto issue = [&](int grp, int c) {
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int cc = c + 32 * u, row = grp * ROWS + r;
                wbuf[u][r] = (cc < nchunks && row < m)
                                 ? load16_any(W + (size_t)row * ldw + (size_t)cc * 16, W, W_end)
                                 : make_uint4(0u, 0u, 0u, 0u);
            }
    };
    if (g < ngroups) issue(g, lane);

    // Digit planes of x_hat (zero past K).
    uint32_t *planes = reinterpret_cast<uint32_t *>(s_planes);
    const int pstride = nchunks * 4;  // words per plane
    for (int q4 = tid; q4 < pstride; q4 += kGemvThreads) {
        uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int k = q4 * 4 + b;
            if (k < K) {
                int d0, d1, d2, d3;
                limb_split(__ldg(xhat + k), d0, d1, d2, d3);
                p0 |= (uint32_t)(d0 & 0xff) << (8 * b);
                p1 |= (uint32_t)(d1 & 0xff) << (8 * b);
                p2 |= (uint32_t)(d2 & 0xff) << (8 * b);
                p3 |= (uint32_t)(d3 & 0xff) << (8 * b);
            }
        }
        planes[q4] = p0;
        planes[pstride + q4] = p1;
        planes[2 * pstride + q4] = p2;
        planes[3 * pstride + q4] = p3;
    }
    __syncthreads();
    const uint4 *P0 = s_planes, *P1 = s_planes + nchunks, *P2 = s_planes + 2 * nchunks,
                *P3 = s_planes + 3 * nchunks;

    for (; g < ngroups; g += gstride) {
        int acc[ROWS][4];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0;

        for (int c = lane; c < nchunks; c += 32 * UNROLL) {
            uint4 cur[UNROLL][ROWS];
#pragma unroll
            for (int u = 0; u < UNROLL; ++u)
#pragma unroll
                for (int r = 0; r < ROWS; ++r) cur[u][r] = wbuf[u][r];
            // prefetch: the next column batch of this group, else the next group
            const int cn = c + 32 * UNROLL;
            if (cn < nchunks) issue(g, cn);
            else if (g + gstride < ngroups) issue(g + gstride, lane);
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int cc = c + 32 * u;
                if (cc < nchunks) {
                    const uint4 l0 = P0[cc], l1 = P1[cc], l2 = P2[cc], l3 = P3[cc];
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const uint4 w = cur[u][r];
                        acc[r][0] = __dp4a((int)w.x, (int)l0.x, acc[r][0]);
                        acc[r][1] = __dp4a((int)w.x, (int)l1.x, acc[r][1]);
                        acc[r][2] = __dp4a((int)w.x, (int)l2.x, acc[r][2]);
                        acc[r][3] = __dp4a((int)w.x, (int)l3.x, acc[r][3]);
                        acc[r][0] = __dp4a((int)w.y, (int)l0.y, acc[r][0]);
                        acc[r][1] = __dp4a((int)w.y, (int)l1.y, acc[r][1]);
                        acc[r][2] = __dp4a((int)w.y, (int)l2.y, acc[r][2]);
                        acc[r][3] = __dp4a((int)w.y, (int)l3.y, acc[r][3]);
                        acc[r][0] = __dp4a((int)w.z, (int)l0.z, acc[r][0]);
                        acc[r][1] = __dp4a((int)w.z, (int)l1.z, acc[r][1]);
                        acc[r][2] = __dp4a((int)w.z, (int)l2.z, acc[r][2]);
                        acc[r][3] = __dp4a((int)w.z, (int)l3.z, acc[r][3]);
                        acc[r][0] = __dp4a((int)w.w, (int)l0.w, acc[r][0]);
                        acc[r][1] = __dp4a((int)w.w, (int)l1.w, acc[r][1]);
                        acc[r][2] = __dp4a((int)w.w, (int)l2.w, acc[r][2]);
                        acc[r][3] = __dp4a((int)w.w, (int)l3.w, acc[r][3]);
                    }
                }
            }
        }

        int v[V];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int p = 0; p < 4; ++p) v[r * 4 + p] = acc[r][p];
        const int tot = transposed_reduce<V>(v, lane);
        // lane l holds entry l / (32/V) = 4 r + p
        constexpr int span = 32 / V;
        const int a1 = __shfl_down_sync(kFull, tot, span);
        const int a2 = __shfl_down_sync(kFull, tot, 2 * span);
        const int a3 = __shfl_down_sync(kFull, tot, 3 * span);
        const int entry = lane / span;
        if ((lane % span) == 0 && (entry & 3) == 0) {
            const int row = g * ROWS + (entry >> 2);
            if (row < m) {
                const int64_t s = (int64_t)tot + ((int64_t)a1 << 8) + ((int64_t)a2 << 16) +
                                  ((int64_t)a3 << 24);
                const uint32_t part = fred_signed(s);
                y[row] = accumulate ? fadd(y[row], part) : part;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Grouped persistent kernel: one launch computes a list of independent batch-1
// products (jobs), each streaming its own matrix once.  One CTA of 512 threads
// per SM (two for large products) takes whole rows: of one job where a few jobs split evenly over the
// CTAs (the rows then run without a break), else an even share of all the
// bytes, job after job.
//
// A thread owns one or two 16-byte chunks of the row (T threads per row, so
// 512 / T rows at a time) and keeps the digits of its columns of x_hat in
// registers.  Its own chunks of M come through a ring of three batches of
// rows in shared memory, filled by its own cp.async (no barrier: only the
// thread that asked for a chunk reads it): 96 KiB in flight per SM, where the
// HBM rate times its latency is about 45.  64 registers and 104 KiB of shared
// memory leave room for the CTAs of the next launch beside these (programmatic
// dependent launch): they fill their ring with M before griddepcontrol.wait
// and only then read x_hat, so the memory system does not drain between
// dependent launches.  M is the server's weight matrix, never written by a
// kernel that signals its dependents early.
//
// Per batch a thread's digit sums are packed in pairs (a0 + 2^8 a1 fits 32
// bits over 8 or 16 lanes), which halves the shuffles of the transposed
// butterfly; 16-bit halves of its results are added in shared memory, and one
// barrier per 256 rows hands them to the threads that reduce mod q and store.
//
// Against a kernel with the digit planes in shared memory, M in registers and
// two CTAs of 128 registers per SM: eight 8B-class layers of four dependent
// launches 402 -> 322 us (5.4 TB/s), 100 requests of 4096 x 4096 252 -> 231
// us (7.3 TB/s); dependent single calls, 4096 x 4096 5.8 -> 4.6 us, 4096 x
// 14336 14.1 -> 12.0, 50000 x 64 15.0 -> 5.0, 256 x 256 2.05 -> 1.9.  Asking
// L2 for more of M before the wait made a token slower (362 -> 378 us and up).
// ---------------------------------------------------------------------------
constexpr int kRingThreads = 512;
constexpr int kRingBatches = 3;  // row batches in flight
constexpr int kRingSlots = 4;    // 16-byte slots per thread and batch
constexpr int kRingSumRows = 16 * (kRingThreads / 32);  // rows per block-wide reduction
constexpr int kRingFewJobs = 8;
constexpr int kRingMinBytes = 16384;  // of M per CTA (1024 x 1024: 2.4 us; 8 KiB 2.8, 64 KiB 2.7)
constexpr long long kRingPairBytes = 256 << 10;  // of M per SM from which an SM takes two CTAs
constexpr int kRingSmem = kRingThreads * kRingBatches * kRingSlots * 16;

template <int NJ>
struct RingArgs {
    int count;
    int split;                // CTAs are split by `first`, else the bytes by `base`
    int first[NJ + 1];        // job j's CTAs are first[j] .. first[j + 1] - 1
    long long base[NJ + 1];   // prefix sums of m_j * K_j
    MvmJob job[NJ];
};

__device__ __forceinline__ void ring_load(uint32_t dst, const int8_t *src) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ring_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void ring_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int CH, int NJ>
__global__ void __launch_bounds__(kRingThreads, 2) k_gemv_ring(const __grid_constant__ RingArgs<NJ> args) {
    extern __shared__ uint4 s_ring[];
    __shared__ __align__(16) int s_sum[2][kRingSumRows][4];
    constexpr int ROWS = kRingSlots / CH;  // rows of a batch
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_ring) + tid * 16u;
    const int cta = (int)blockIdx.x;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    static_assert(2 * kRingSumRows == kRingThreads, "one row of sums per thread to clear");
    reinterpret_cast<int4 *>(s_sum)[tid] = make_int4(0, 0, 0, 0);
    __syncthreads();
    // the first job of this CTA
    long long lo = 0, hi = 0;
    int j = 0;
    if (args.split) {
        while (cta >= args.first[j + 1]) ++j;
    } else {
        const long long total = args.base[args.count];
        lo = total * cta / gridDim.x;
        hi = total * (cta + 1) / gridDim.x;
        int last = args.count - 1;
        while (j < last) {
            const int mid = (j + last) / 2;
            if (args.base[mid + 1] > lo) last = mid; else j = mid + 1;
        }
    }
    bool waited = false;
    int buf = 0;

    for (bool more = true; more && j < args.count; ++j) {
        const MvmJob &job = args.job[j];
        const int K = job.K, nchunks = K / 16;
        int row_a, row_b;
        if (args.split) {
            const uint32_t n = (uint32_t)(args.first[j + 1] - args.first[j]), i = (uint32_t)(cta - args.first[j]);
            row_a = (int)((uint32_t)job.m * i / n);
            row_b = (int)((uint32_t)job.m * (i + 1) / n);
            more = false;
        } else {
            // rows whose first byte lies in [lo, hi)
            const long long b0 = args.base[j];
            row_a = lo > b0 ? (int)((lo - b0 + K - 1) / K) : 0;
            row_b = (int)min((long long)job.m, (hi - b0 + K - 1) / K);
            more = args.base[j + 1] < hi;
        }
        if (row_a >= row_b) continue;
        int T = 32;  // threads per row
        while (T < kRingThreads && T * CH < nchunks) T *= 2;
        const int G = kRingThreads / T, grp = tid / T, ct = tid % T;
        const int per = (row_b - row_a + G - 1) / G;  // rows of a group (the same for all groups)

        const int8_t *src = job.W + (size_t)(row_a + grp) * job.ldw + (size_t)ct * 16;
        const size_t step = (size_t)G * job.ldw;
        const int mine = (row_b - row_a - grp + G - 1) / G;  // rows of this group (0 or less: none)
        int next = 0;                                        // the next row to load
        auto load = [&](uint32_t at) {                       // a batch of rows into the slots at `at`
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                if (next + r < mine) {
#pragma unroll
                    for (int i = 0; i < CH; ++i)
                        if (ct + i * T < nchunks)
                            ring_load(at + (uint32_t)((r * CH + i) * kRingThreads * 16), src + (size_t)i * T * 16);
                }
                src += step;
            }
            ring_commit();
            next += ROWS;
        };
        constexpr uint32_t kBatchBytes = kRingSlots * kRingThreads * 16;
#pragma unroll
        for (int d = 0; d < kRingBatches; ++d) load(ring + d * kBatchBytes);
        if (!waited) {
            // x_hat may only be read after the wait; L2 may fetch it before
            // (eight 8B-class layers 338.5 -> 334.7 us)
#pragma unroll
            for (int i = 0; i < CH; ++i)
                if (grp == 0 && ct + i * T < nchunks)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(job.xhat + (size_t)(ct + i * T) * 16));
            asm volatile("griddepcontrol.wait;" ::: "memory");
            waited = true;
        }
        uint32_t dig[CH][4][4];
#pragma unroll
        for (int i = 0; i < CH; ++i) {
#pragma unroll
            for (int q = 0; q < 4; ++q) dig[i][0][q] = dig[i][1][q] = dig[i][2][q] = dig[i][3][q] = 0u;
            if (ct + i * T < nchunks) {
                const uint4 *xp = reinterpret_cast<const uint4 *>(job.xhat + (size_t)(ct + i * T) * 16);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 xv = xp[q];  // written while this kernel was in place already: no read-only load
                    const uint32_t xs[4] = {xv.x, xv.y, xv.z, xv.w};
                    uint32_t u[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) u[e] = ((xs[e] > kHalfQ ? xs[e] - kQ : xs[e]) + 0x80808080u) ^ 0x80808080u;
                    // 4 x 4 byte transpose: plane p holds byte p of the four
                    const uint32_t a = __byte_perm(u[0], u[1], 0x5140), b = __byte_perm(u[2], u[3], 0x5140);
                    const uint32_t c = __byte_perm(u[0], u[1], 0x7362), d = __byte_perm(u[2], u[3], 0x7362);
                    dig[i][0][q] = __byte_perm(a, b, 0x5410);
                    dig[i][1][q] = __byte_perm(a, b, 0x7632);
                    dig[i][2][q] = __byte_perm(c, d, 0x5410);
                    dig[i][3][q] = __byte_perm(c, d, 0x7632);
                }
            }
        }

        uint32_t at = 0;
        const int blk = kRingSumRows / G;  // rows of a group per block-wide reduction (a multiple of ROWS)
        for (int i0 = 0; i0 < per; i0 += blk) {
            const int i1 = min(per, i0 + blk);
            for (int i = i0; i < i1; i += ROWS) {
                ring_wait<kRingBatches - 1>();
                const uint4 *rp = s_ring + at * (kRingSlots * kRingThreads) + tid;
                // v[2 r] = a0 + 2^8 a1, v[2 r + 1] = a2 + 2^8 a3 of row r
                int v[2 * ROWS];
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) {
                        const uint4 w = rp[(r * CH + ch) * kRingThreads];
                        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            a0 = __dp4a((int)ww[q], (int)dig[ch][0][q], a0);
                            a1 = __dp4a((int)ww[q], (int)dig[ch][1][q], a1);
                            a2 = __dp4a((int)ww[q], (int)dig[ch][2][q], a2);
                            a3 = __dp4a((int)ww[q], (int)dig[ch][3][q], a3);
                        }
                    }
                    v[2 * r] = a0 + a1 * 256;
                    v[2 * r + 1] = a2 + a3 * 256;
                }
                load(ring + at * kBatchBytes);
                at = at + 1 == kRingBatches ? 0u : at + 1;
                // each lane ends with one entry summed over 16 / CH lanes:
                // |a| <= 2^18 CH, so the sum stays below 2^30 + 2^22
                constexpr int V = 2 * ROWS;
#pragma unroll
                for (int n = V, o = 16; n > 1; n >>= 1, o >>= 1) {
                    const bool upper = (lane & o) != 0;
#pragma unroll
                    for (int e = 0; e < n / 2; ++e) {
                        const int send = upper ? v[e] : v[e + n / 2];
                        const int keep = upper ? v[e + n / 2] : v[e];
                        v[e] = keep + __shfl_xor_sync(kFull, send, o);
                    }
                }
                constexpr int kSpan = 32 / V;  // lanes that hold parts of one entry
                v[0] += __shfl_xor_sync(kFull, v[0], kSpan / 2);
                if ((lane & (kSpan / 2)) == 0) {
                    const int e = lane / kSpan;
                    int *sp = &s_sum[buf][(i - i0 + (e >> 1)) * G + grp][2 * (e & 1)];
                    atomicAdd(sp, v[0] & 0xffff);
                    atomicAdd(sp + 1, v[0] >> 16);
                }
            }
            __syncthreads();
            // the other buffer takes the next block's sums meanwhile
            for (int e = tid; e < (i1 - i0 + ROWS - 1) / ROWS * ROWS * G; e += kRingThreads) {
                int *sp = s_sum[buf][e];
                const int64_t sum = (int64_t)sp[0] + ((int64_t)(sp[1] + sp[2]) << 16) + ((int64_t)sp[3] << 32);
                sp[0] = sp[1] = sp[2] = sp[3] = 0;
                const int row = row_a + i0 * G + e;
                if (row < row_b) {
                    const uint32_t part = fred_signed(sum);
                    job.y[row] = job.accumulate ? fadd(job.y[row], part) : part;
                }
            }
            buf ^= 1;
        }
        ring_wait<0>();
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int CH, int NJ>
cudaError_t run_gemv_ring(const MvmJob *jobs, int count, cudaStream_t s) {
    RingArgs<NJ> args;
    args.count = count;
    args.base[0] = 0;
    long long rows = 0;
    for (int j = 0; j < count; ++j) {
        args.job[j] = jobs[j];
        args.base[j + 1] = args.base[j] + (long long)jobs[j].m * jobs[j].K;
        rows += jobs[j].m;
    }
    if (rows == 0) return cudaSuccess;
    const auto kern = k_gemv_ring<CH, NJ>;
    const cudaError_t attr = func_attr((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingSmem);
    if (attr != cudaSuccess) return attr;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // One CTA per SM where every CTA gets enough of M, so that the next
    // launch's fill their rings beside it; two for a few jobs that are large.
    // Two are placed evenly whatever ran before (every slot of an SM takes
    // one), one need not be: a launch that comes while the one before it ends,
    // as the second after a pause does, puts two CTAs on the SMs that are
    // empty, and the launches that depend on it inherit that (a token through
    // eight 8B-class layers after a pause: 356 or 485 us by turns, now 348; back
    // to back 346 -> 336).  Below the line the rings hold much of the share
    // and the overlap is worth more (dependent single calls, two CTAs against
    // one: 8192 x 4096 8.3 and 6.8 us, 6144 x 6144 8.0 and 7.6; above it
    // 8192 x 8192 11.0 and 11.6, gate and up of 14336 x 4096 17.3 and 18.7;
    // 100 requests 249 and 237).  4096 x 14336 pays 1.1 us for the even
    // placement that the gate and up after it depend on (12.0 and 10.9): its
    // 13 rows of 14 KiB a CTA leave a ring of two chunks little to run on.
    const long long total = args.base[count];
    const long long slots = count <= kRingFewJobs && total >= sms * kRingPairBytes ? 2LL * sms : sms;
    const int grid = (int)std::max(1LL, std::min({slots, rows, total / kRingMinBytes}));
    args.split = 0;
    if (count <= kRingFewJobs && count * 8 <= grid) {
        // CTAs for each job, where that splits the bytes within 12 % of evenly
        // (q, k, v of an 8B-class layer: 7.6 -> 6.0 us; a CTA that goes from
        // one job to the next drains its ring)
        double worst = 0;
        int at = 0;
        bool fits = true;
        for (int j = 0; j < count; ++j) {
            args.first[j] = at;
            at = j + 1 == count ? grid : (int)((double)args.base[j + 1] * grid / total + 0.5);
            const int n = at - args.first[j];
            fits = fits && n >= 1 && (long long)jobs[j].m * (n + 1) < (1LL << 32);
            if (n >= 1) worst = std::max(worst, (double)((jobs[j].m + n - 1) / n) * jobs[j].K);
        }
        args.first[count] = grid;
        if (fits && worst * grid <= 1.12 * (double)total + 16384.0 * grid) args.split = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(kRingThreads, 1, 1);
    cfg.dynamicSmemBytes = kRingSmem;
    cfg.stream = s;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 1;
    return counted_launch(cudaLaunchKernelEx(&cfg, kern, args));
}

// One launch for up to kMultiMaxJobs jobs of K <= kMultiMaxK.
cudaError_t run_gemv_multi(const MvmJob *jobs, int count, cudaStream_t s) {
    int kmax = 16;
    for (int j = 0; j < count; ++j) kmax = std::max(kmax, jobs[j].K);
    // one chunk per thread while a row's chunks fit the CTA, else two; few
    // jobs in a small parameter block (a launch copies the whole block)
    if (kmax <= 16 * kRingThreads)
        return count <= kRingFewJobs ? run_gemv_ring<1, kRingFewJobs>(jobs, count, s)
                                     : run_gemv_ring<1, kMultiMaxJobs>(jobs, count, s);
    return count <= kRingFewJobs ? run_gemv_ring<2, kRingFewJobs>(jobs, count, s)
                                 : run_gemv_ring<2, kMultiMaxJobs>(jobs, count, s);
}

template <int ROWS, int UNROLL>
cudaError_t run_gemv(const int8_t *W, size_t ldw, int m, int K, const uint32_t *xhat, uint32_t *y,
                     bool accumulate, cudaStream_t s) {
    const int nchunks = (K + 15) / 16;
    const size_t smem = (size_t)nchunks * 16 * 4;
    auto kern = k_gemv<ROWS, UNROLL>;
    // set once (outside any stream capture that a later call might be part of)
    const cudaError_t attr = func_attr((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kGemvMaxK * 4);
    if (attr != cudaSuccess) return attr;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int ngroups = (m + ROWS - 1) / ROWS;
    const int grid = ngroups < sms ? ngroups : sms;
    kern<<<grid, kGemvThreads, smem, s>>>(W, ldw, m, K, xhat, y, accumulate); note_launch();
    return cudaGetLastError();
}

}  // namespace

bool multi_eligible(const MvmJob &j) {
    return j.K % 16 == 0 && j.ldw % 16 == 0 && (reinterpret_cast<uintptr_t>(j.W) & 15u) == 0 &&
           (reinterpret_cast<uintptr_t>(j.xhat) & 15u) == 0;
}

cudaError_t launch_gemv_multi(const MvmJob *jobs, int count, cudaStream_t s) {
    // Jobs with K beyond one shared-memory segment are split into K segments;
    // segment k of every job goes into launch k, later launches accumulate.
    std::vector<MvmJob> seg;
    for (int k0 = 0;; k0 += kMultiMaxK) {
        seg.clear();
        for (int j = 0; j < count; ++j) {
            if (jobs[j].K <= k0) continue;
            MvmJob t = jobs[j];
            t.W = jobs[j].W + k0;
            t.xhat = jobs[j].xhat + k0;
            t.K = jobs[j].K - k0 < kMultiMaxK ? jobs[j].K - k0 : kMultiMaxK;
            t.accumulate = k0 > 0 ? 1 : jobs[j].accumulate;
            seg.push_back(t);
        }
        if (seg.empty()) return cudaSuccess;
        for (size_t a = 0; a < seg.size(); a += kMultiMaxJobs) {
            const int n = (int)std::min(seg.size() - a, (size_t)kMultiMaxJobs);
            cudaError_t e = run_gemv_multi(seg.data() + a, n, s);
            if (e != cudaSuccess) return e;
        }
    }
}

cudaError_t launch_gemv(const int8_t *W, int m, int K, const uint32_t *xhat, uint32_t *y,
                        uint32_t *err, cudaStream_t s) {
    (void)err;
    if (m <= 0 || K <= 0) return cudaSuccess;
    MvmJob j{W, xhat, y, m, K, (size_t)K, 0};
    if (multi_eligible(j)) return launch_gemv_multi(&j, 1, s);
    for (int k0 = 0; k0 < K; k0 += kGemvMaxK) {
        const int kl = K - k0 < kGemvMaxK ? K - k0 : kGemvMaxK;
        cudaError_t e = run_gemv<2, 2>(W + k0, (size_t)K, m, kl, xhat + k0, y, k0 > 0, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace pv
