// C ABI of the pvMVMD library (include/pvmvmd.h): parameter resolution, the
// host's sampler of the public RAA codes (contexts sample theirs on the
// device), context management, and the ordering of the device kernels for each
// protocol call.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <initializer_list>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "common.cuh"
#include "launch.h"

namespace pv {

// The library's device error word (kErr* bits).
__device__ uint32_t g_error_word = 0;

namespace {

// Domain tags of the ChaCha20 nonces (tag, index): the two codes, the masks
// and the challenges each read their own keystream.
constexpr uint32_t kTagCodeX = 1;       // G_x: pi1 = 1, pi2 = 2, v1 = 3, v2 = 4
constexpr uint32_t kTagCodeY = 5;       // G_y: pi1 = 5, pi2 = 6, v1 = 7, v2 = 8
static_assert(kTagCodeY == kTagCodeX + 4, "code `which` reads tags kTagCodeX + 4 which + 0..3");
constexpr uint32_t kTagMask = 9;
constexpr uint32_t kTagChallenge = 10;
constexpr uint32_t kTagBvPrimary = 21;    // batch verification challenges
constexpr uint32_t kTagBvSecondary = 22;
// Encode batches of at least this many vectors as the lanes of N x B arrays
// (launch_lane_syndrome) when the code does not fit one CTA's shared memory and
// the sliced kernel does not take them.
constexpr int kLaneMinBatch = 32;
// Server products of at most this many vectors use the small-batch paths.
constexpr int kSmallBatchMax = 16;

// --------------------------------------------------------------------------
// Host ChaCha20 keystream (RFC 8439 Sec. 2.3) read as 32-bit words.
// --------------------------------------------------------------------------
class KeyStream {
  public:
    KeyStream(const pvmvmd_key &key, uint32_t tag, uint64_t index) : key_(key) {
        nonce_[0] = tag;
        nonce_[1] = (uint32_t)index;
        nonce_[2] = (uint32_t)(index >> 32);
    }
    uint32_t word() {
        if (used_ == 16) refill();
        return block_[used_++];
    }
    // Uniform in [0, k): top bitlen(k-1) bits, rejected while >= k.
    uint32_t below(uint32_t k) {
        if (k <= 1) return 0;
        int bits = 0;
        for (uint32_t v = k - 1; v; v >>= 1) ++bits;
        for (;;) {
            const uint32_t v = word() >> (32 - bits);
            if (v < k) return v;
        }
    }
    // Uniform in F* = [1, q): top 31 bits, rejected outside [1, q).
    uint32_t nonzero_field() {
        for (;;) {
            const uint32_t v = word() >> 1;
            if (v != 0 && v < kQ) return v;
        }
    }

  private:
    static uint32_t rotl(uint32_t v, int c) { return (v << c) | (v >> (32 - c)); }
    static void quarter(uint32_t *s, int a, int b, int c, int d) {
        s[a] += s[b]; s[d] = rotl(s[d] ^ s[a], 16);
        s[c] += s[d]; s[b] = rotl(s[b] ^ s[c], 12);
        s[a] += s[b]; s[d] = rotl(s[d] ^ s[a], 8);
        s[c] += s[d]; s[b] = rotl(s[b] ^ s[c], 7);
    }
    void refill() {
        uint32_t in[16] = {0x61707865u, 0x3320646eu, 0x79622d32u, 0x6b206574u};
        std::memcpy(in + 4, key_.k, sizeof key_.k);
        in[12] = counter_++;
        in[13] = nonce_[0];
        in[14] = nonce_[1];
        in[15] = nonce_[2];
        uint32_t s[16];
        std::memcpy(s, in, sizeof s);
        for (int i = 0; i < 10; ++i) {
            quarter(s, 0, 4, 8, 12); quarter(s, 1, 5, 9, 13);
            quarter(s, 2, 6, 10, 14); quarter(s, 3, 7, 11, 15);
            quarter(s, 0, 5, 10, 15); quarter(s, 1, 6, 11, 12);
            quarter(s, 2, 7, 8, 13); quarter(s, 3, 4, 9, 14);
        }
        for (int i = 0; i < 16; ++i) block_[i] = s[i] + in[i];
        used_ = 0;
    }
    pvmvmd_key key_;
    uint32_t nonce_[3];
    uint32_t counter_ = 0;
    uint32_t block_[16];
    int used_ = 16;
};

void sample_code_host(const pvmvmd_key &key, int which, uint32_t N, uint32_t *pi1, uint32_t *pi2,
                      uint32_t *v1, uint32_t *v2) {
    // code `which` reads tags 4 which + 1 .. 4 which + 4 (G_x = 0, G_y = 1;
    // the batch verification codes are 3 and 4)
    const uint32_t tag0 = kTagCodeX + 4u * (uint32_t)which;
    uint32_t *perms[2] = {pi1, pi2};
    for (int p = 0; p < 2; ++p) {  // Fisher-Yates, last index first
        KeyStream ks(key, tag0 + p, 0);
        uint32_t *a = perms[p];
        for (uint32_t i = 0; i < N; ++i) a[i] = i;
        for (uint32_t i = N; i-- > 1;) {
            const uint32_t j = ks.below(i + 1);
            const uint32_t tmp = a[i];
            a[i] = a[j];
            a[j] = tmp;
        }
    }
    uint32_t *scales[2] = {v1, v2};
    for (int p = 0; p < 2; ++p) {
        KeyStream ks(key, tag0 + 2 + p, 0);
        for (uint32_t i = 0; i < N; ++i) scales[p][i] = ks.nonzero_field();
    }
}

// --------------------------------------------------------------------------
// Device helpers
// --------------------------------------------------------------------------
int check_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PVMVMD_E_NODEVICE;
    int major = 0, minor = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
        return PVMVMD_E_NODEVICE;
    return (major == 10 && minor == 3) ? PVMVMD_OK : PVMVMD_E_NODEVICE;
}

std::atomic<unsigned long long> g_kernel_launches{0};
unsigned long long kernel_launches() { return g_kernel_launches.load(std::memory_order_relaxed); }
}  // namespace
void note_launch() { g_kernel_launches.fetch_add(1, std::memory_order_relaxed); }
namespace {
int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

uint32_t *error_word() {
    static std::mutex mu;
    static uint32_t *addr[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_error_word) != cudaSuccess) return nullptr;
        addr[dev] = static_cast<uint32_t *>(p);
    }
    return addr[dev];
}

#define PV_CUDA(expr)                                  \
    do {                                               \
        cudaError_t e_ = (expr);                       \
        if (e_ != cudaSuccess) {                       \
            (void)cudaGetLastError();                  \
            return e_ == cudaErrorMemoryAllocation ? PVMVMD_E_NOMEM : PVMVMD_E_CUDA; \
        }                                              \
    } while (0)

template <typename T>
cudaError_t dev_alloc(T **p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
}

struct CodeDev {
    uint32_t *pi1 = nullptr, *pi2 = nullptr, *v1 = nullptr, *v2 = nullptr;
    uint32_t *pi1inv = nullptr, *pi2inv = nullptr, *v2p = nullptr;
    uint32_t *v2m = nullptr, *v1pm = nullptr;  // Montgomery-scaled v2 and v1 o pi1^-1
    uint32_t *v1m = nullptr;                   // Montgomery-scaled v1
    uint32_t *slices = nullptr;                // the sliced syndrome's tables (G_x, where it is used)
};

}  // namespace
}  // namespace pv

struct pvmvmd_ctx {
    int device = 0;
    pvmvmd_params params{};
    int m = 0, K = 0, rate = 0, Nx = 0, Ny = 0, t_x = 0, t_y = 0, ell = 0, sb = 0;
    pv::CodeDev gx, gy;
    uint32_t *PT = nullptr, *Q = nullptr;
    uint32_t *F = nullptr, *Fy = nullptr, *chal = nullptr, *g = nullptr, *u = nullptr;
    // scan status words of the encode (status) and of the challenges
    // (status_y): an encode and a decode share no scratch
    unsigned long long *status = nullptr, *status_y = nullptr;
    // lane-parallel encode scratch (null when scratch_batch < kLaneMinBatch)
    uint32_t *S = nullptr, *laux = nullptr;
    // decode: the challenge kernels run on `side` (highest stream priority),
    // forked from and joined back to the caller's stream, while the decrypt
    // streams P^T
    cudaStream_t side = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    uint32_t *sync = nullptr;  // of the one-kernel decode
    // the last verification ran on a caller's stream; a call was captured
    bool on_caller = false, captured = false;
    std::vector<void *> owned;
};

// Batch verification (Protocol 2) for B matrices of one shape m x n.
struct pvmvmd_bv_ctx {
    int device = 0;
    int B = 0, m = 0, n = 0, rate = 0, N = 0, N2 = 0, t = 0, ell = 0, t2 = 0, ell2 = 0;
    pv::CodeDev g, g2;       // primary code (dimension m), secondary code (dimension B n)
    uint32_t *Qs = nullptr;    // N x B n: row i = (Q_1[i], ..., Q_B[i]) = Qt^T (public)
    uint32_t *QauxT = nullptr; // N' x N: Qaux transposed
    uint32_t *Yt = nullptr, *Z = nullptr;  // m x B, N x B
    uint32_t *chal2 = nullptr, *R = nullptr, *F2 = nullptr;
    uint32_t *eS = nullptr;                      // encode scratch: S
    unsigned long long *estatus = nullptr;       // and scan status words
    unsigned long long *status = nullptr;
    std::vector<void *> owned;
};

namespace pv {
namespace {

template <typename Ctx, typename T>
cudaError_t ctx_alloc(Ctx *c, T **p, size_t count) {
    cudaError_t e = dev_alloc(p, count);
    if (e == cudaSuccess) c->owned.push_back(*p);
    return e;
}

// Samples the context's two codes (numbers which[k], lengths N[k]) on the device,
// their tables in one allocation.  Enqueued on s: the scratch is freed by the
// caller once the stream has drained.
template <typename Ctx>
int sample_codes(Ctx *c, const pvmvmd_key &key, CodeDev *const code[2], const int which[2], const uint32_t N[2],
                 uint32_t **scratch, cudaStream_t s) {
    size_t words = 0, swords = 0;
    auto up = [](size_t n) { return (n + 63) & ~(size_t)63; };  // tables start on 256-byte boundaries
    for (int k = 0; k < 2; ++k) {
        words += 10 * up(N[k]);
        swords += up(code_draw_scratch_words(N[k]));
    }
    uint32_t *t = nullptr;
    PV_CUDA(ctx_alloc(c, &t, words));
    PV_CUDA(dev_alloc(scratch, swords));
    CodeDraws draws[2];
    uint32_t *sc[2], *at = *scratch;
    for (int k = 0; k < 2; ++k) {
        CodeDev &d = *code[k];
        for (uint32_t **p : {&d.pi1, &d.pi2, &d.v1, &d.v2, &d.pi1inv, &d.pi2inv, &d.v2p, &d.v2m, &d.v1pm, &d.v1m}) {
            *p = t;
            t += up(N[k]);
        }
        // code `which` reads tags kTagCodeX + 4 which + 0 .. 3
        draws[k] = CodeDraws{N[k], kTagCodeX + 4u * (uint32_t)which[k], d.pi1, d.pi2, d.v1, d.v2, d.pi1inv, d.pi2inv,
                             d.v2p, d.v2m, d.v1pm, d.v1m, {}};
        sc[k] = at;
        at += up(code_draw_scratch_words(N[k]));
    }
    PV_CUDA(launch_code_draws(key, draws, 2, sc, s));
    return PVMVMD_OK;
}

// Y (N x L lanes, row stride ldy) = G^T applied to the L lanes of X (n x L,
// row stride ldx; row i holds message entry i of every lane), in lane chunks.
// One chunk of lanes with caller-provided scratch (S: N x nl; status:
// encode_scan_status_words(N, nl) 64-bit words); no
// allocation, no sync.
int encode_lanes_into(const CodeDev &d, uint32_t n, uint32_t r, const void *X, bool x_is_i8, size_t ldx,
                      uint32_t nl, uint32_t *Y, size_t ldy, uint32_t *S, unsigned long long *status,
                      uint32_t *err, cudaStream_t s) {
    const uint32_t N = n * r;
    cudaError_t e = encode_scan_clear(status, N, nl, s);
    if (e == cudaSuccess)  // S = A^T V1 Pi1^T R^T X
        e = launch_encode_scan(X, x_is_i8, ldx, d.pi1, r, d.v1m, N, nl, S, nl, status, err, s);
    if (e == cudaSuccess) e = encode_scan_clear(status, N, nl, s);
    if (e == cudaSuccess)  // Y = A^T V2 Pi2^T S
        e = launch_encode_scan(S, false, nl, d.pi2, 1, d.v2m, N, nl, Y, ldy, status, err, s);
    return e == cudaSuccess ? PVMVMD_OK : PVMVMD_E_CUDA;
}

// Scratch of encode_lanes, allocated once for all the encodings of a
// preprocessing (a 512 MiB cudaMalloc and cudaFree take 0.44 ms).
struct LaneScratch {
    uint32_t *S = nullptr;
    unsigned long long *status = nullptr;
    ~LaneScratch() {
        cudaFree(S);
        cudaFree(status);
    }
    // lanes per chunk: about 256 MiB of S (at 4096 x 4096 0.1 ms less to
    // allocate and free than 512 MiB, at the same speed), 2048 lanes up to 1 GiB
    static size_t lanes(uint32_t N, uint32_t L) {
        const size_t few = ((size_t)1 << 26) / N, most = ((size_t)1 << 28) / N;
        size_t lc = std::max(few, std::min<size_t>(2048, most)) / 256 * 256;
        if (lc < 256) lc = 256;
        return lc < L ? lc : L;
    }
    // for encodings of length N[k] over L[k] lanes
    int alloc(std::initializer_list<std::pair<uint32_t, uint32_t>> uses) {
        size_t s = 0, w = 0;
        for (const auto &u : uses) {
            const size_t lc = lanes(u.first, u.second);
            s = std::max(s, (size_t)u.first * lc);
            w = std::max(w, encode_scan_status_words(u.first, (uint32_t)lc));
        }
        return dev_alloc(&S, s) == cudaSuccess && dev_alloc(&status, w) == cudaSuccess
                   ? PVMVMD_OK
                   : PVMVMD_E_NOMEM;
    }
};

// Y (N x L lanes, row stride ldy) = G^T applied to the L lanes of X (n x L,
// row stride ldx; row i holds message entry i of every lane; int8 or
// uint32), in lane chunks (preprocessing only).
int encode_lanes(const CodeDev &d, uint32_t n, uint32_t r, const void *X, bool x_is_i8, size_t ldx,
                 uint32_t L, uint32_t *Y, size_t ldy, const LaneScratch &sc, uint32_t *err, cudaStream_t s) {
    const size_t lc = LaneScratch::lanes(n * r, L);
    for (uint32_t l0 = 0; l0 < L; l0 += (uint32_t)lc) {
        const uint32_t nl = (uint32_t)((L - l0) < lc ? (L - l0) : lc);
        const void *Xl = x_is_i8 ? static_cast<const void *>(static_cast<const int8_t *>(X) + l0)
                                 : static_cast<const void *>(static_cast<const uint32_t *>(X) + l0);
        const int st = encode_lanes_into(d, n, r, Xl, x_is_i8, ldx, nl, Y + l0, ldy, sc.S, sc.status, err, s);
        if (st != PVMVMD_OK) return st;
    }
    return PVMVMD_OK;
}

int read_and_clear_error() {
    uint32_t *ew = error_word();
    if (!ew) return PVMVMD_E_CUDA;
    uint32_t v = 0;
    if (cudaMemcpy(&v, ew, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return PVMVMD_E_CUDA;
    if (v) {
        const uint32_t zero = 0;
        if (cudaMemcpy(ew, &zero, 4, cudaMemcpyHostToDevice) != cudaSuccess) return PVMVMD_E_CUDA;
        return PVMVMD_E_DEVICE_TIMEOUT;
    }
    return PVMVMD_OK;
}

}  // namespace

uint32_t *library_error_word() { return error_word(); }

namespace {
std::mutex g_debug_mu;
DebugWait g_debug;
}  // namespace

DebugWait debug_wait() {
    std::lock_guard<std::mutex> lock(g_debug_mu);
    return g_debug;
}

}  // namespace pv

using namespace pv;

extern "C" {

const char *pvmvmd_strerror(int status) {
    switch (status) {
        case PVMVMD_OK: return "success";
        case PVMVMD_E_ARG: return "invalid argument (null pointer or bad value)";
        case PVMVMD_E_SHAPE: return "shape or batch size outside the supported range";
        case PVMVMD_E_PARAM: return "inconsistent protocol parameters (e.g. t > N)";
        case PVMVMD_E_CUDA: return "a CUDA runtime call or kernel launch failed";
        case PVMVMD_E_NOMEM: return "out of memory";
        case PVMVMD_E_DEVICE_TIMEOUT: return "a bounded device-side wait expired";
        case PVMVMD_E_NODEVICE: return "no sm_103 (GB300) CUDA device is current";
        default: return "unknown status";
    }
}

int pvmvmd_params_resolve(const pvmvmd_params *in, int m, int K, pvmvmd_params *out) {
    if (!out || m < 1 || K < 1) return PVMVMD_E_ARG;
    pvmvmd_params p{};
    if (in) p = *in;
    if (p.lambda < 0 || p.kappa < 0 || p.rate < 0 || p.delta < 0 || p.t_x < 0 || p.t_y < 0 ||
        p.ell < 0 || p.scratch_batch < 0 || p.delta >= 1.0)
        return PVMVMD_E_PARAM;
    if (p.lambda == 0) p.lambda = 128;
    if (p.kappa == 0) p.kappa = 40;
    if (p.rate == 0) p.rate = 8;
    if (p.delta == 0) p.delta = 0.5;
    if (p.scratch_batch == 0) p.scratch_batch = 64;
    const double Nx = (double)p.rate * K, Ny = (double)p.rate * m;
    if (Nx > 4294967295.0 || Ny > 4294967295.0) return PVMVMD_E_SHAPE;
    if (p.t_x == 0) {  // Eq. (1)
        const double t = std::ceil(std::log(2.0) * ((double)p.lambda - std::log2(Nx)) / p.delta);
        p.t_x = t < 1 ? 1 : (int)t;
    }
    // Thm 5.2, by the two cases of its proof: with lf = log2(|F| - 1),
    // case 1 (lf >= kappa + 1) needs (1-delta)^t <= 2^-(kappa+1) and ell = 1;
    // case 2 needs (1-delta)^t <= 1/(|F|-1) and ell = ceil(kappa / (lf - 1)).
    const double lf = std::log2((double)(kQ - 1));
    const double per = -std::log2(1.0 - p.delta);
    const bool case1 = lf >= p.kappa + 1;
    if (p.t_y == 0) p.t_y = (int)std::ceil((case1 ? (double)(p.kappa + 1) : lf) / per);
    if (p.ell == 0) p.ell = case1 ? 1 : (int)std::ceil((double)p.kappa / (lf - 1.0));
    if (p.t_x > Nx || p.t_y > Ny || p.t_x > PVMVMD_MAX_T || p.t_y > PVMVMD_MAX_T || p.ell > 16 ||
        p.ell < 1)
        return PVMVMD_E_PARAM;
    *out = p;
    return PVMVMD_OK;
}

int pvmvmd_code_sample_host(const pvmvmd_key *key, int which, uint32_t N, uint32_t *pi1,
                            uint32_t *pi2, uint32_t *v1, uint32_t *v2) {
    if (!key || !pi1 || !pi2 || !v1 || !v2 || (which != 0 && which != 1)) return PVMVMD_E_ARG;
    sample_code_host(*key, which, N, pi1, pi2, v1, v2);
    return PVMVMD_OK;
}

void pvmvmd_destroy(pvmvmd_ctx *ctx) {
    if (!ctx) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(ctx->device);
    for (void *p : ctx->owned) cudaFree(p);
    if (ctx->fork) cudaEventDestroy(ctx->fork);
    if (ctx->join) cudaEventDestroy(ctx->join);
    if (ctx->side) cudaStreamDestroy(ctx->side);
    cudaSetDevice(cur);
    delete ctx;
}

namespace pv {
namespace {
int preprocess_impl(const void *W_dev, bool w16, int m, int K, const pvmvmd_params *params,
                    const pvmvmd_key *key, void *stream, pvmvmd_ctx **out);
}  // namespace
}  // namespace pv

int pvmvmd_preprocess(const int8_t *W_dev, int m, int K, const pvmvmd_params *params,
                      const pvmvmd_key *key, void *stream, pvmvmd_ctx **out) {
    return pv::preprocess_impl(W_dev, false, m, K, params, key, stream, out);
}

int pvmvmd_preprocess_i16(const int16_t *W_dev, int m, int K, const pvmvmd_params *params,
                          const pvmvmd_key *key, void *stream, pvmvmd_ctx **out) {
    return pv::preprocess_impl(W_dev, true, m, K, params, key, stream, out);
}

namespace pv {
namespace {
int preprocess_impl(const void *W_dev, bool w16, int m, int K, const pvmvmd_params *params,
                    const pvmvmd_key *key, void *stream, pvmvmd_ctx **out) {
    if (!out) return PVMVMD_E_ARG;
    *out = nullptr;
    if (!W_dev || !key) return PVMVMD_E_ARG;
    if (m < 1 || K < 1 || K > PVMVMD_MAX_K) return PVMVMD_E_SHAPE;
    int st = check_device();
    if (st) return st;
    pvmvmd_params p;
    st = pvmvmd_params_resolve(params, m, K, &p);
    if (st) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;

    pvmvmd_ctx *c = new (std::nothrow) pvmvmd_ctx();
    if (!c) return PVMVMD_E_NOMEM;
    cudaGetDevice(&c->device);
    c->params = p;
    c->m = m;
    c->K = K;
    c->rate = p.rate;
    c->Nx = p.rate * K;
    c->Ny = p.rate * m;
    c->t_x = p.t_x;
    c->t_y = p.t_y;
    c->ell = p.ell;
    c->sb = p.scratch_batch;

    auto fail = [&](int code) {
        cudaStreamSynchronize(s);  // what is enqueued may still use the context
        (void)cudaGetLastError();
        pvmvmd_destroy(c);
        return code;
    };
    // temporaries: freed on every way out, once the stream has drained (the
    // context's own memory too, where the call fails)
    struct Temp {
        uint32_t *draws = nullptr, *M32 = nullptr, *MT32 = nullptr;
        int8_t *MT = nullptr;
        LaneScratch lanes;
        cudaStream_t s;
        ~Temp() {
            cudaStreamSynchronize(s);
            cudaFree(draws);
            cudaFree(M32);
            cudaFree(MT32);
            cudaFree(MT);
        }
    } tmp;
    tmp.s = s;
    CodeDev *const codes[2] = {&c->gx, &c->gy};
    const int which[2] = {0, 1};
    const uint32_t lengths[2] = {(uint32_t)c->Nx, (uint32_t)c->Ny};
    if ((st = sample_codes(c, *key, codes, which, lengths, &tmp.draws, s))) return fail(st);
    if (!syndrome_fused_fits(c->Nx, c->t_x) && syndrome_sliced_fits(c->Nx, K, c->rate, c->t_x)) {
        CodeDev &d = c->gx;
        if (ctx_alloc(c, &d.slices, slice_table_words(c->Nx)) != cudaSuccess) return fail(PVMVMD_E_NOMEM);
        if (launch_slice_tables(d.pi1, d.pi2, d.v2m, c->Nx, c->rate, d.slices, s) != cudaSuccess)
            return fail(PVMVMD_E_CUDA);
    }
    // the small arrays in one allocation
    const size_t f = (size_t)((c->sb + 3) & ~3) * c->Nx;  // lanes padded to 4
    const bool lanes = c->sb >= kLaneMinBatch;
    uint32_t *small = nullptr;
    size_t words = 0;
    auto take = [&](size_t n) {  // on 256-byte boundaries
        const size_t at = words;
        words += (n + 63) & ~(size_t)63;
        return at;
    };
    const size_t oF = take(f), oFy = take((size_t)c->ell * c->Ny), ochal = take((size_t)c->ell * 2 * c->t_y),
                 og = take((size_t)c->ell * m), ou = take((size_t)c->ell * K),
                 ostatus = take(2 * scan_status_words(c->Nx, c->sb)),
                 ostatus_y = take(2 * scan_status_words(c->Ny, c->ell)), osync = take(kDecodeSyncWords),
                 oS = take(lanes ? lane_state_words(c->t_x, c->sb) : 0),
                 olaux = take(lanes ? lane_aux_words(c->Nx, c->sb) : 0);
    if (ctx_alloc(c, &small, words) != cudaSuccess || ctx_alloc(c, &c->PT, (size_t)c->Nx * m) != cudaSuccess ||
        ctx_alloc(c, &c->Q, (size_t)c->Ny * K) != cudaSuccess)
        return fail(PVMVMD_E_NOMEM);
    c->F = small + oF;
    c->Fy = small + oFy;
    c->chal = small + ochal;
    c->g = small + og;
    c->u = small + ou;
    c->status = reinterpret_cast<unsigned long long *>(small + ostatus);
    c->status_y = reinterpret_cast<unsigned long long *>(small + ostatus_y);
    c->sync = small + osync;
    if (lanes) {
        c->S = small + oS;
        c->laux = small + olaux;
    }
    // the tiled syndrome and the one-kernel decode find these zero and leave them so
    if (cudaMemsetAsync(c->sync, 0, kDecodeSyncWords * sizeof(uint32_t), s) != cudaSuccess ||
        cudaMemsetAsync(c->status, 0, scan_status_words(c->Nx, c->sb) * sizeof(unsigned long long), s) != cudaSuccess ||
        cudaMemsetAsync(c->status_y, 0, scan_status_words(c->Ny, c->ell) * sizeof(unsigned long long), s) !=
            cudaSuccess)
        return fail(PVMVMD_E_CUDA);
    // the challenge kernels are few and short; at the highest priority their
    // blocks take SMs as the decrypt's blocks drain instead of queueing
    // behind the rest of the decrypt's grid
    int prio_least = 0, prio_greatest = 0;
    if (cudaDeviceGetStreamPriorityRange(&prio_least, &prio_greatest) != cudaSuccess ||
        cudaStreamCreateWithPriority(&c->side, cudaStreamNonBlocking, prio_greatest) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->join, cudaEventDisableTiming) != cudaSuccess)
        return fail(PVMVMD_E_CUDA);
    if ((st = tmp.lanes.alloc({{(uint32_t)c->Nx, (uint32_t)m}, {(uint32_t)c->Ny, (uint32_t)K}}))) return fail(st);
    const void *rows = W_dev, *cols = nullptr;  // M by rows (lanes: its columns) and transposed
    if (w16) {
        // 16-bit M: lift it to F_q, then encode as uint32 lanes
        if (dev_alloc(&tmp.M32, (size_t)m * K) != cudaSuccess || dev_alloc(&tmp.MT32, (size_t)m * K) != cudaSuccess)
            return fail(PVMVMD_E_NOMEM);
        if (launch_lift_i16(static_cast<const int16_t *>(W_dev), (size_t)m * K, tmp.M32, s) != cudaSuccess ||
            launch_transpose_u32(tmp.M32, m, K, tmp.MT32, s) != cudaSuccess)
            return fail(PVMVMD_E_CUDA);
        rows = tmp.M32;
        cols = tmp.MT32;
    } else {
        if (dev_alloc(&tmp.MT, (size_t)m * K) != cudaSuccess) return fail(PVMVMD_E_NOMEM);
        if (launch_transpose_i8(static_cast<const int8_t *>(W_dev), m, K, tmp.MT, s) != cudaSuccess)
            return fail(PVMVMD_E_CUDA);
        cols = tmp.MT;
    }
    // P^T = G_x^T M^T: the m rows of M are the lanes; Q = G_y^T M: its K columns
    st = encode_lanes(c->gx, K, c->rate, cols, !w16, (size_t)m, m, c->PT, (size_t)m, tmp.lanes, err, s);
    if (!st) st = encode_lanes(c->gy, m, c->rate, rows, !w16, (size_t)K, K, c->Q, (size_t)K, tmp.lanes, err, s);
    if (!st && cudaStreamSynchronize(s) != cudaSuccess) st = PVMVMD_E_CUDA;
    if (!st) st = read_and_clear_error();
    if (st) return fail(st);
    *out = c;
    return PVMVMD_OK;
}
}  // namespace
}  // namespace pv

int pvmvmd_weights_split_i16(const int16_t *W_dev, int m, int K, int8_t *Whi_dev, int8_t *Wlo_dev,
                             void *stream) {
    using namespace pv;
    if (!W_dev || !Whi_dev || !Wlo_dev) return PVMVMD_E_ARG;
    if (m < 1 || K < 1) return PVMVMD_E_SHAPE;
    PV_CUDA(launch_split_i16(W_dev, (size_t)m * K, Whi_dev, Wlo_dev, static_cast<cudaStream_t>(stream)));
    return PVMVMD_OK;
}

namespace pv {
namespace {
// The paths of a product of 2 <= B <= 16 vectors: one pass over M per four
// vectors with dp4a, or the tensor-core product with 16-vector tiles (8 to 10 us
// until M is large) from 12 MiB of M passed over that way.  GEMV against
// tensor cores, us: 4096 x 2560 with 4 vectors 8.2 and 8.7, with 8 12.8 and
// 9.2; 1024 x 4096 with 8 8.2 and 8.7, with 12 11.4 and 8.7; 4096 x 4096 with 2
// 10.6 and 9.7; 14336 x 4096 with 4 23.6 and 15.4.  Both planes of a 16-bit
// M: 4096 x 2560 with 4 12.8 and 12.8, with 8 20.0 and 12.4; 4096 x 4096 with 2
// 17.0 and 13.8.  Where the scratch of the tensor-core product cannot be had
// (memory, or a stream under capture that has not run as large a call), the
// GEMV's smaller one serves.
bool small_batch_ok(const void *W, int K, const uint32_t *Xhat, int B) {
    return B > 1 && B <= kSmallBatchMax && K % 16 == 0 &&
           ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(Xhat)) & 15u) == 0;
}
bool small_batch_on_tensor(int m, int K, int B) {
    return (double)m * K * ((B + 3) / 4) >= 12.0 * 1024 * 1024;
}
}  // namespace
}  // namespace pv

// Both planes in one launch: of the small-batch kernel, which combines them
// itself (4096 x 2560, 4 vectors: 18.9 -> 12.8 us a call), as two jobs of the
// grouped tensor-core product (8 vectors: 28.8 -> 12.4; under capture only if its
// scratch is there already) or of the batch-1 kernel (one vector: 28.6 ->
// 17.5 us).
int pvmvmd_server_mvm_i16(const int8_t *Whi_dev, const int8_t *Wlo_dev, int m, int K, const uint32_t *Xhat_dev,
                          int B, uint32_t *Yhat_dev, uint32_t *Ytmp_dev, void *stream) {
    using namespace pv;
    if (!Whi_dev || !Wlo_dev || !Ytmp_dev || !Xhat_dev || !Yhat_dev) return PVMVMD_E_ARG;
    if (m < 1 || K < 1 || K > PVMVMD_MAX_K || B < 1) return PVMVMD_E_SHAPE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (small_batch_ok(Whi_dev, K, Xhat_dev, B) && small_batch_ok(Wlo_dev, K, Xhat_dev, B)) {
        if (small_batch_on_tensor(m, K, B)) {
            uint32_t *err = error_word();
            if (!err) return PVMVMD_E_CUDA;
            const BatchJob jobs[2] = {{Whi_dev, Xhat_dev, Yhat_dev, m, K, B}, {Wlo_dev, Xhat_dev, Ytmp_dev, m, K, B}};
            const cudaError_t e = launch_batched_grouped(jobs, 2, err, s, true);
            if (e == cudaSuccess) PV_CUDA(launch_combine_256(Yhat_dev, Ytmp_dev, (size_t)B * m, s));
            if (e != cudaErrorNotReady && e != cudaErrorMemoryAllocation) {
                PV_CUDA(e);
                return PVMVMD_OK;
            }
            (void)cudaGetLastError();
        }
        PV_CUDA(launch_gemv_small_batch(Wlo_dev, m, K, Xhat_dev, B, Yhat_dev, s, Whi_dev));
        return PVMVMD_OK;
    }
    if (B == 1) {
        const pvmvmd_mvm_job jobs[2] = {{Whi_dev, Xhat_dev, Yhat_dev, m, K}, {Wlo_dev, Xhat_dev, Ytmp_dev, m, K}};
        const int st = pvmvmd_server_mvm_multi(jobs, 2, stream);
        if (st) return st;
    } else {
        int st = pvmvmd_server_mvm(Whi_dev, m, K, Xhat_dev, B, Yhat_dev, stream);
        if (!st) st = pvmvmd_server_mvm(Wlo_dev, m, K, Xhat_dev, B, Ytmp_dev, stream);
        if (st) return st;
    }
    PV_CUDA(launch_combine_256(Yhat_dev, Ytmp_dev, (size_t)B * m, s));
    return PVMVMD_OK;
}

int pvmvmd_state_size(const pvmvmd_ctx *ctx, int B, size_t *bytes) {
    if (!ctx || !bytes || B < 0) return PVMVMD_E_ARG;
    *bytes = (size_t)B * 2 * ctx->t_x * sizeof(uint32_t);
    return PVMVMD_OK;
}

namespace pv {
namespace {
// Xhat = X + G_x e_x for the B vectors (X null: Xhat = G_x e_x alone).
int encode_batch(pvmvmd_ctx *ctx, const uint32_t *X_dev, int B, const pvmvmd_key *key,
                 uint32_t *Xhat_dev, void *st_dev, cudaStream_t s);
}  // namespace
}  // namespace pv

int pvmvmd_encode(pvmvmd_ctx *ctx, const uint32_t *X_dev, int B, const pvmvmd_key *key,
                  uint32_t *Xhat_dev, void *st_dev, void *stream) {
    if (!ctx || !X_dev || !key || !Xhat_dev || !st_dev) return PVMVMD_E_ARG;
    if (B < 1) return PVMVMD_E_SHAPE;
    return pv::encode_batch(ctx, X_dev, B, key, Xhat_dev, st_dev, static_cast<cudaStream_t>(stream));
}

int pvmvmd_boost_prepare(pvmvmd_ctx *ctx, int B, const pvmvmd_key *key, uint32_t *mask_in_dev,
                         uint32_t *mask_out_dev, void *st_dev, void *stream) {
    using namespace pv;
    if (!ctx || !key || !mask_in_dev || !mask_out_dev || !st_dev) return PVMVMD_E_ARG;
    if (B < 1) return PVMVMD_E_SHAPE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int st = encode_batch(ctx, nullptr, B, key, mask_in_dev, st_dev, s);
    if (st != PVMVMD_OK) return st;
    PV_CUDA(launch_output_mask(ctx->PT, ctx->m, static_cast<const uint32_t *>(st_dev), ctx->t_x, B,
                               mask_out_dev, s));
    return PVMVMD_OK;
}

int pvmvmd_boost_encode(const uint32_t *X_dev, const uint32_t *mask_in_dev, int B, int K,
                        uint32_t *Xhat_dev, void *stream) {
    using namespace pv;
    if (!X_dev || !mask_in_dev || !Xhat_dev) return PVMVMD_E_ARG;
    if (B < 1 || K < 1) return PVMVMD_E_SHAPE;
    PV_CUDA(launch_field_add(X_dev, mask_in_dev, (size_t)B * K, Xhat_dev,
                             static_cast<cudaStream_t>(stream)));
    return PVMVMD_OK;
}

namespace pv {
namespace {
int encode_batch(pvmvmd_ctx *ctx, const uint32_t *X_dev, int B, const pvmvmd_key *key,
                 uint32_t *Xhat_dev, void *st_dev, cudaStream_t s) {
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    uint32_t *stp = static_cast<uint32_t *>(st_dev);
    const CodeDev &d = ctx->gx;
    const bool fits = syndrome_fused_fits(ctx->Nx, ctx->t_x);
    const bool lanes = B >= kLaneMinBatch && ctx->laux && !fits;
    const bool tiles = syndrome_tiles_eligible((uint32_t)ctx->t_x);
    const uint32_t ntiles = scan_tiles((uint32_t)ctx->Nx);
    // A code too long for that: a CTA per vector, two per SM, slice by slice.
    //  * Against the lanes, back to back and alone (one encode and a field add,
    //    about 8 us of it launches): K = 8192, B = 256: 55 against 83 us and 71
    //    against 85; B = 100: 23 / 45 and 44 / 46; B = 64: 15 / 40 but 44 / 42;
    //    K = 5700, B = 32: 7 / 36 and 36 / 37; K = 13000, B = 152: 54 / 97 and
    //    74 / 99, B = 128: 47 / 68 but 74 / 70.  The lines keep both.
    //  * Against the tiles, whose every CTA draws the whole support, so that a
    //    call costs B N_x t_x where it costs N_x here: the line is where one call
    //    alone takes about as long (back to back and alone): t_x = 333, B = 16:
    //    K = 5700: 7.9 against 27 us and 50 against 46, K = 8192: 9.2 / 31 and 57 /
    //    48, K = 10000: 12 / 49 and 70 / 71; t_x = 156, B = 31: K = 5700: 8.9 / 29
    //    and 47 / 49, K = 8192: 11 / 36 and 55 / 51, K = 13000: 18 / 58 but 84 / 74.
    //  * Where the scratch holds fewer vectors than the batch has, or the tiles
    //    do not take the support: K = 8192, 16 vectors one by one 64 / 104.
    bool sliced = false;
    if (d.slices && lanes)
        sliced = B >= (ctx->Nx <= 48 * 1024 ? kLaneMinBatch : ctx->Nx <= 80 * 1024 ? 2 * sm_count() / 3 : sm_count());
    else if (d.slices)
        sliced = !tiles || B > ctx->sb || (uint64_t)B * ctx->t_x > (uint64_t)33 * sm_count();
    if (sliced) {
        PV_CUDA(launch_syndrome_sliced(*key, kTagMask, 0, ctx->Nx, ctx->t_x, (uint32_t)B, d.slices, d.v1m, ctx->K, stp,
                                       X_dev, Xhat_dev, s));
        return PVMVMD_OK;
    }
    if (lanes) {
        // vectors as lanes: every permutation step moves whole rows (a code
        // that fits one CTA's shared memory stays on chip in the fused kernel)
        for (int b0 = 0; b0 < B; b0 += ctx->sb) {
            const uint32_t L = (uint32_t)(B - b0 < ctx->sb ? B - b0 : ctx->sb);
            PV_CUDA(launch_lane_syndrome(*key, kTagMask, (uint64_t)b0, ctx->Nx, ctx->t_x, L, d.pi2,
                                         d.v2m, d.v1m, d.pi1inv, ctx->K, ctx->rate,
                                         stp + (size_t)b0 * 2 * ctx->t_x, ctx->S, ctx->F, ctx->laux,
                                         X_dev ? X_dev + (size_t)b0 * ctx->K : nullptr,
                                         Xhat_dev + (size_t)b0 * ctx->K, s));
        }
        return PVMVMD_OK;
    }
    // A code of more than four tiles (more where the support is long, since each
    // draws it by itself) and a batch of at most one tile per SM:
    // small CTAs, one per tile, finish sooner than a CTA per vector.  Measured
    // (one encode and a field add, graph replay, about 8 us of it launches):
    // K = 4096, B = 8: 16.8 against 25.2 us; K = 2560, B = 8: 17.6 against
    // 21.4; K = 1001 (four tiles), B = 1: 13.7 and 13.7; t_x = 335, B = 1, alone:
    // K = 4096 32.5 against 34, K = 2048 (eight tiles) 33 against 28; back to back the two
    // tie at one tile per SM (K = 4096, B = 8: 7.1 against 6.7 us a call) and
    // beyond it the CTA per vector wins (B = 16: 12.1 against 6.7).  It needs no
    // scratch either: a batch of more vectors than the scratch holds stays whole.
    const bool spread = tiles && ntiles > 4 && 32 * ntiles > (uint32_t)ctx->t_x && B <= ctx->sb &&
                        (uint64_t)B * ntiles <= (uint64_t)sm_count();
    if (fits && !spread) {
        // sample, scan and gather in one launch per batch, no scratch
        PV_CUDA(launch_syndrome_fused(*key, kTagMask, 0, ctx->Nx, ctx->t_x, (uint32_t)B, d.pi1inv, d.pi2,
                                      d.v2m, d.v1pm, ctx->K, ctx->rate, stp, X_dev, Xhat_dev, s));
        return PVMVMD_OK;
    }
    if (tiles) {
        for (int b0 = 0; b0 < B; b0 += ctx->sb) {
            const uint32_t nb = (uint32_t)(B - b0 < ctx->sb ? B - b0 : ctx->sb);
            PV_CUDA(launch_syndrome_tiles(*key, kTagMask, (uint64_t)b0, ctx->Nx, ctx->t_x, nb, d.pi2inv, d.v2p,
                                          d.v1m, d.pi1inv, ctx->K, ctx->rate, stp + (size_t)b0 * 2 * ctx->t_x,
                                          ctx->F, ctx->status, err,
                                          X_dev ? X_dev + (size_t)b0 * ctx->K : nullptr,
                                          Xhat_dev + (size_t)b0 * ctx->K, s, /*pdl=*/true));
        }
        return PVMVMD_OK;
    }
    for (int b0 = 0; b0 < B; b0 += ctx->sb) {
        const uint32_t nb = (uint32_t)(B - b0 < ctx->sb ? B - b0 : ctx->sb);
        uint32_t *e = stp + (size_t)b0 * 2 * ctx->t_x;
        PV_CUDA(launch_sample_sparse(*key, kTagMask, (uint64_t)b0, ctx->Nx, ctx->t_x, nb, e,
                                     ctx->status, scan_status_words(ctx->Nx, nb), s));
        PV_CUDA(launch_syndrome_scan(d.pi2inv, d.v2p, d.v1, ctx->Nx, e, ctx->t_x, nb, ctx->F,
                                     ctx->status, err, s));
        PV_CUDA(launch_syndrome_gather(d.pi1inv, ctx->K, ctx->rate, ctx->F, ctx->Nx,
                                       X_dev ? X_dev + (size_t)b0 * ctx->K : nullptr,
                                       Xhat_dev + (size_t)b0 * ctx->K, nb, s));
    }
    return PVMVMD_OK;
}
}  // namespace
}  // namespace pv

int pvmvmd_server_mvm(const int8_t *W_dev, int m, int K, const uint32_t *Xhat_dev, int B,
                      uint32_t *Yhat_dev, void *stream) {
    if (!W_dev || !Xhat_dev || !Yhat_dev) return PVMVMD_E_ARG;
    if (m < 1 || K < 1 || K > PVMVMD_MAX_K || B < 1) return PVMVMD_E_SHAPE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    if (B == 1) {
        PV_CUDA(launch_gemv(W_dev, m, K, Xhat_dev, Yhat_dev, err, s));
        return PVMVMD_OK;
    }
    if (small_batch_ok(W_dev, K, Xhat_dev, B)) {
        if (small_batch_on_tensor(m, K, B)) {
            const BatchJob job{W_dev, Xhat_dev, Yhat_dev, m, K, B};
            const cudaError_t e = launch_batched_grouped(&job, 1, err, s, true);
            if (e != cudaErrorNotReady && e != cudaErrorMemoryAllocation) {
                PV_CUDA(e);
                return PVMVMD_OK;
            }
            (void)cudaGetLastError();
        }
        PV_CUDA(launch_gemv_small_batch(W_dev, m, K, Xhat_dev, B, Yhat_dev, s));
        return PVMVMD_OK;
    }
    PV_CUDA(launch_batched(W_dev, m, K, Xhat_dev, B, Yhat_dev, err, s));
    return PVMVMD_OK;
}

int pvmvmd_server_mvm_multi(const pvmvmd_mvm_job *jobs, int count, void *stream) {
    if (!jobs || count < 1) return count < 1 ? PVMVMD_E_SHAPE : PVMVMD_E_ARG;
    for (int i = 0; i < count; ++i) {
        const pvmvmd_mvm_job &j = jobs[i];
        if (!j.W_dev || !j.xhat_dev || !j.yhat_dev) return PVMVMD_E_ARG;
        if (j.m < 1 || j.K < 1 || j.K > PVMVMD_MAX_K) return PVMVMD_E_SHAPE;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    std::vector<MvmJob> grouped;
    grouped.reserve(count);
    for (int i = 0; i < count; ++i) {
        const pvmvmd_mvm_job &j = jobs[i];
        MvmJob t{j.W_dev, j.xhat_dev, j.yhat_dev, j.m, j.K, (size_t)j.K, 0};
        if (multi_eligible(t))
            grouped.push_back(t);
        else
            PV_CUDA(launch_gemv(j.W_dev, j.m, j.K, j.xhat_dev, j.yhat_dev, err, s));
    }
    if (!grouped.empty()) PV_CUDA(launch_gemv_multi(grouped.data(), (int)grouped.size(), s));
    return PVMVMD_OK;
}

int pvmvmd_server_mvm_grouped(const pvmvmd_mvm_batch_job *jobs, int count, void *stream) {
    if (!jobs || count < 1) return count < 1 ? PVMVMD_E_SHAPE : PVMVMD_E_ARG;
    for (int i = 0; i < count; ++i) {
        const pvmvmd_mvm_batch_job &j = jobs[i];
        if (!j.W_dev || !j.Xhat_dev || !j.Yhat_dev) return PVMVMD_E_ARG;
        if (j.m < 1 || j.K < 1 || j.K > PVMVMD_MAX_K || j.B < 1) return PVMVMD_E_SHAPE;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    // the tensor-core products together in one persistent launch; every
    // other job takes the path pvmvmd_server_mvm gives it
    std::vector<BatchJob> grouped;
    std::vector<MvmJob> single;
    for (int i = 0; i < count; ++i) {
        const pvmvmd_mvm_batch_job &j = jobs[i];
        if (j.B > 1 && batched_grouped_eligible(j.W_dev, j.Xhat_dev, j.m, j.K, j.B)) {
            grouped.push_back(BatchJob{j.W_dev, j.Xhat_dev, j.Yhat_dev, j.m, j.K, j.B});
            continue;
        }
        if (j.B == 1) {
            MvmJob t{j.W_dev, j.Xhat_dev, j.Yhat_dev, j.m, j.K, (size_t)j.K, 0};
            if (multi_eligible(t)) {
                single.push_back(t);
                continue;
            }
        }
        const int st = pvmvmd_server_mvm(j.W_dev, j.m, j.K, j.Xhat_dev, j.B, j.Yhat_dev, stream);
        if (st != PVMVMD_OK) return st;
    }
    if (!single.empty()) PV_CUDA(launch_gemv_multi(single.data(), (int)single.size(), s));
    if (!grouped.empty()) PV_CUDA(launch_batched_grouped(grouped.data(), (int)grouped.size(), err, s));
    return PVMVMD_OK;
}

namespace pv {
namespace {
// The challenges of a call: e_q <- E_{t_y}^{N_y}, shared by its vectors, and
// g_q = G_y e_q, u_q = e_q^T Q from them, on stream cs.  They rest on the key and
// the context alone.
int challenge_chain(pvmvmd_ctx *ctx, const pvmvmd_key *challenge_key, cudaStream_t cs) {
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    const CodeDev &d = ctx->gy;
    if (syndrome_tiles_eligible((uint32_t)ctx->t_y)) {
        PV_CUDA(launch_syndrome_tiles(*challenge_key, kTagChallenge, 0, ctx->Ny, ctx->t_y, (uint32_t)ctx->ell,
                                      d.pi2inv, d.v2p, d.v1m, d.pi1inv, ctx->m, ctx->rate, nullptr, ctx->Fy,
                                      ctx->status_y, err, nullptr, ctx->g, cs, false, ctx->Q, ctx->K, ctx->u));
    } else {
        PV_CUDA(launch_sample_sparse(*challenge_key, kTagChallenge, 0, ctx->Ny, ctx->t_y, ctx->ell,
                                     ctx->chal, ctx->status_y, scan_status_words(ctx->Ny, ctx->ell), cs));
        PV_CUDA(launch_syndrome_scan(d.pi2inv, d.v2p, d.v1, ctx->Ny, ctx->chal, ctx->t_y, ctx->ell,
                                     ctx->Fy, ctx->status_y, err, cs));
        PV_CUDA(launch_syndrome_gather(d.pi1inv, ctx->m, ctx->rate, ctx->Fy, ctx->Ny, nullptr, ctx->g,
                                       ctx->ell, cs));
        PV_CUDA(launch_verify_u(ctx->Q, ctx->K, ctx->chal, ctx->t_y, ctx->ell, ctx->u, cs));
    }
    return PVMVMD_OK;
}

bool overlaps(const void *a, const void *b, size_t bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + bytes && y < x + bytes;
}

// The verification on the context's side stream, the decrypt on s, joined.
int decode_beside(pvmvmd_ctx *ctx, const void *st_dev, const uint32_t *mask_out_dev, const uint32_t *Xhat_dev,
                  const uint32_t *Yhat_dev, int B, const pvmvmd_key *challenge_key, uint32_t *Y_dev,
                  int32_t *accept_dev, cudaStream_t s) {
    const bool early = !ctx->captured && !ctx->on_caller;
    int st = PVMVMD_OK;
    if (early && (st = challenge_chain(ctx, challenge_key, ctx->side))) return st;
    PV_CUDA(cudaEventRecord(ctx->fork, s));
    PV_CUDA(cudaStreamWaitEvent(ctx->side, ctx->fork, 0));
    if (!early && (st = challenge_chain(ctx, challenge_key, ctx->side))) return st;
    ctx->on_caller = false;
    PV_CUDA(launch_check(Xhat_dev, ctx->K, Yhat_dev, ctx->m, ctx->g, ctx->u, (uint32_t)ctx->ell, B, accept_dev,
                         ctx->side));
    PV_CUDA(launch_decrypt(ctx->PT, ctx->m, static_cast<const uint32_t *>(st_dev), ctx->t_x, (uint32_t)ctx->Nx,
                           Yhat_dev, B, Y_dev, s, mask_out_dev));
    PV_CUDA(cudaEventRecord(ctx->join, ctx->side));
    PV_CUDA(cudaStreamWaitEvent(s, ctx->join, 0));
    return PVMVMD_OK;
}

// Verify and decrypt: Y = Yhat - P e_x from st, or Y = Yhat - mask_out when
// mask_out is given (boost mode).
//  * A large decrypt: one kernel on the caller's stream (launch_decode).
//  * Else the verification runs on the context's side stream while the
//    decrypt runs on the caller's, which then waits for the side stream.
//    Only the check reads what the caller's stream produced, so only it waits
//    for that stream: the challenges are formed while, say, the server's
//    product still runs (round trip of 1030 x 1001, 70 vectors 36.5 -> 29 us).
//    Their scratch is free by then, since every earlier verification ran on
//    the side stream too -- or on a caller's stream, as a replay of a captured
//    call also does: then they wait as well.
//  * When Y overwrites Yhat the verification must read Yhat first, and both
//    run in order on the caller's stream.
int decode_verify_batch(pvmvmd_ctx *ctx, const void *st_dev, const uint32_t *mask_out_dev,
                        const uint32_t *Xhat_dev, const uint32_t *Yhat_dev, int B,
                        const pvmvmd_key *challenge_key, uint32_t *Y_dev, int32_t *accept_dev,
                        cudaStream_t s) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {  // the legacy stream, while another is captured
        (void)cudaGetLastError();
        capture = cudaStreamCaptureStatusActive;
    }
    if (capture != cudaStreamCaptureStatusNone) ctx->captured = true;
    const bool in_place = overlaps(Y_dev, Yhat_dev, (size_t)B * ctx->m * sizeof(uint32_t));
    if (!in_place && !mask_out_dev && decode_wins(ctx->m, B, ctx->t_x, ctx->t_y, ctx->ell)) {
        uint32_t *err = error_word();
        if (!err) return PVMVMD_E_CUDA;
        const CodeDev &d = ctx->gy;
        const DecodeCall c{*challenge_key, kTagChallenge, (uint32_t)ctx->Ny, (uint32_t)ctx->t_y, (uint32_t)ctx->ell,
                           (uint32_t)ctx->rate, (uint32_t)ctx->t_x, (uint32_t)ctx->Nx, d.pi2inv, d.v2p, d.v1m,
                           d.pi1inv, ctx->Fy, ctx->status_y, err, ctx->sync, ctx->Q, ctx->u, ctx->g, ctx->PT,
                           static_cast<const uint32_t *>(st_dev), Xhat_dev, Yhat_dev, Y_dev, accept_dev, ctx->m,
                           ctx->K, B};
        // the side stream's last use of the scratch was joined to the
        // caller's stream by the call that made it
        ctx->on_caller = true;
        PV_CUDA(launch_decode(c, s));
        return PVMVMD_OK;
    }
    if (!in_place) {
        const int st = decode_beside(ctx, st_dev, mask_out_dev, Xhat_dev, Yhat_dev, B, challenge_key, Y_dev,
                                     accept_dev, s);
        // not joined: what the side stream has of the call must not run beside
        // the next one, which may use the scratch on another stream
        if (st != PVMVMD_OK && capture == cudaStreamCaptureStatusNone) {
            cudaStreamSynchronize(ctx->side);
            (void)cudaGetLastError();
        }
        return st;
    }
    ctx->on_caller = true;
    const int st = challenge_chain(ctx, challenge_key, s);
    if (st) return st;
    PV_CUDA(launch_check(Xhat_dev, ctx->K, Yhat_dev, ctx->m, ctx->g, ctx->u, (uint32_t)ctx->ell, B, accept_dev, s));
    PV_CUDA(launch_decrypt(ctx->PT, ctx->m, static_cast<const uint32_t *>(st_dev), ctx->t_x, (uint32_t)ctx->Nx,
                           Yhat_dev, B, Y_dev, s, mask_out_dev));
    return PVMVMD_OK;
}
}  // namespace
}  // namespace pv

int pvmvmd_decode_verify(pvmvmd_ctx *ctx, const void *st_dev, const uint32_t *Xhat_dev,
                         const uint32_t *Yhat_dev, int B, const pvmvmd_key *challenge_key,
                         uint32_t *Y_dev, int32_t *accept_dev, void *stream) {
    if (!ctx || !st_dev || !Xhat_dev || !Yhat_dev || !challenge_key || !Y_dev || !accept_dev)
        return PVMVMD_E_ARG;
    if (B < 1) return PVMVMD_E_SHAPE;
    return pv::decode_verify_batch(ctx, st_dev, nullptr, Xhat_dev, Yhat_dev, B, challenge_key, Y_dev,
                                   accept_dev, static_cast<cudaStream_t>(stream));
}

int pvmvmd_boost_decode_verify(pvmvmd_ctx *ctx, const uint32_t *mask_out_dev,
                               const uint32_t *Xhat_dev, const uint32_t *Yhat_dev, int B,
                               const pvmvmd_key *challenge_key, uint32_t *Y_dev,
                               int32_t *accept_dev, void *stream) {
    if (!ctx || !mask_out_dev || !Xhat_dev || !Yhat_dev || !challenge_key || !Y_dev || !accept_dev)
        return PVMVMD_E_ARG;
    if (B < 1) return PVMVMD_E_SHAPE;
    return pv::decode_verify_batch(ctx, nullptr, mask_out_dev, Xhat_dev, Yhat_dev, B, challenge_key,
                                   Y_dev, accept_dev, static_cast<cudaStream_t>(stream));
}

namespace pv {
namespace {
// Scratch of pvmvmd_code_encode_lanes: S (N x L), the scan's 64-bit status
// words, each at a 16-byte aligned offset.
struct EncodeScratch {
    size_t s_off, status_off, bytes;
};
EncodeScratch encode_scratch_layout(uint32_t N, uint32_t L) {
    auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    EncodeScratch e;
    e.s_off = 0;
    e.status_off = up((size_t)N * L * 4);
    e.bytes = e.status_off + up(encode_scan_status_words(N, L) * 8);
    return e;
}
}  // namespace
}  // namespace pv

int pvmvmd_code_encode_scratch(const pvmvmd_ctx *ctx, int which, int L, size_t *bytes) {
    if (!ctx || !bytes || (which != 0 && which != 1)) return PVMVMD_E_ARG;
    if (L < 1) return PVMVMD_E_SHAPE;
    const uint32_t N = which == 0 ? ctx->Nx : ctx->Ny;
    *bytes = pv::encode_scratch_layout(N, (uint32_t)L).bytes;
    return PVMVMD_OK;
}

int pvmvmd_code_encode_lanes(const pvmvmd_ctx *ctx, int which, const uint32_t *X_dev, int L,
                             uint32_t *Y_dev, void *scratch_dev, void *stream) {
    using namespace pv;
    if (!ctx || !X_dev || !Y_dev || !scratch_dev || (which != 0 && which != 1)) return PVMVMD_E_ARG;
    if (L < 1) return PVMVMD_E_SHAPE;
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    const CodeDev &d = which == 0 ? ctx->gx : ctx->gy;
    const uint32_t n = which == 0 ? (uint32_t)ctx->K : (uint32_t)ctx->m;
    const EncodeScratch lay = encode_scratch_layout(n * (uint32_t)ctx->rate, (uint32_t)L);
    uint8_t *base = static_cast<uint8_t *>(scratch_dev);
    return encode_lanes_into(d, n, (uint32_t)ctx->rate, X_dev, false, (size_t)L, (uint32_t)L, Y_dev, (size_t)L,
                             reinterpret_cast<uint32_t *>(base + lay.s_off),
                             reinterpret_cast<unsigned long long *>(base + lay.status_off), err,
                             static_cast<cudaStream_t>(stream));
}

int pvmvmd_debug_expire_wait(int site, uint32_t index, uint64_t limit) {
    if (site != PVMVMD_DEBUG_WAIT_OFF && site != PVMVMD_DEBUG_WAIT_SCAN && site != PVMVMD_DEBUG_WAIT_PRODUCT)
        return PVMVMD_E_ARG;
    if (site != PVMVMD_DEBUG_WAIT_OFF && limit == 0) return PVMVMD_E_ARG;
    std::lock_guard<std::mutex> lock(g_debug_mu);
    g_debug.site = site;
    g_debug.index = site == PVMVMD_DEBUG_WAIT_OFF ? 0u : index;
    g_debug.limit = site == PVMVMD_DEBUG_WAIT_OFF ? 0u : limit;
    return PVMVMD_OK;
}

unsigned long long pvmvmd_kernel_launches(void) { return pv::kernel_launches(); }

int pvmvmd_device_status(void *stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) {
        (void)cudaGetLastError();
        return PVMVMD_E_CUDA;
    }
    return read_and_clear_error();
}

int pvmvmd_ctx_info(const pvmvmd_ctx *ctx, pvmvmd_ctx_view *v) {
    if (!ctx || !v) return PVMVMD_E_ARG;
    v->m = ctx->m;
    v->K = ctx->K;
    v->rate = ctx->rate;
    v->N_x = ctx->Nx;
    v->N_y = ctx->Ny;
    v->t_x = ctx->t_x;
    v->t_y = ctx->t_y;
    v->ell = ctx->ell;
    v->gx_pi1 = ctx->gx.pi1;
    v->gx_pi2 = ctx->gx.pi2;
    v->gx_v1 = ctx->gx.v1;
    v->gx_v2 = ctx->gx.v2;
    v->gy_pi1 = ctx->gy.pi1;
    v->gy_pi2 = ctx->gy.pi2;
    v->gy_v1 = ctx->gy.v1;
    v->gy_v2 = ctx->gy.v2;
    v->PT = ctx->PT;
    v->Q = ctx->Q;
    return PVMVMD_OK;
}

}  // extern "C"


// ---------------------------------------------------------------------------
// Batch verification, Protocol 2
// ---------------------------------------------------------------------------
void pvmvmd_bv_destroy(pvmvmd_bv_ctx *ctx) {
    if (!ctx) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(ctx->device);
    for (void *p : ctx->owned) cudaFree(p);
    cudaSetDevice(cur);
    delete ctx;
}

int pvmvmd_bv_preprocess(const int8_t *W_dev, int B, int m, int n, const pvmvmd_bv_params *params,
                         const pvmvmd_key *key, void *stream, pvmvmd_bv_ctx **out) {
    using namespace pv;
    if (!out) return PVMVMD_E_ARG;
    *out = nullptr;
    if (!W_dev || !key) return PVMVMD_E_ARG;
    if (B < 1 || m < 1 || n < 1) return PVMVMD_E_SHAPE;
    const int rate = params && params->rate ? params->rate : 8;
    const long long N = (long long)rate * m, N2 = (long long)rate * B * n;
    // the device sampler holds a bitmap of N bits in shared memory
    if (rate < 2 || N > 8LL * PVMVMD_MAX_K || N2 > 8LL * PVMVMD_MAX_K) return PVMVMD_E_SHAPE;
    const int t = params && params->t ? params->t : 31, ell = params && params->ell ? params->ell : 2;
    const int t2 = params && params->t2 ? params->t2 : 31, ell2 = params && params->ell2 ? params->ell2 : 2;
    if (t < 1 || ell < 1 || t2 < 1 || ell2 < 1 || t > N || t2 > N2) return PVMVMD_E_PARAM;
    int st = check_device();
    if (st) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    pvmvmd_bv_ctx *c = new (std::nothrow) pvmvmd_bv_ctx();
    if (!c) return PVMVMD_E_NOMEM;
    cudaGetDevice(&c->device);
    c->B = B; c->m = m; c->n = n; c->rate = rate; c->N = (int)N; c->N2 = (int)N2;
    c->t = t; c->ell = ell; c->t2 = t2; c->ell2 = ell2;
    auto fail = [&](int code) {
        cudaStreamSynchronize(s);
        (void)cudaGetLastError();
        pvmvmd_bv_destroy(c);
        return code;
    };
    const uint32_t Bn = (uint32_t)B * n;
    struct Temp {
        uint32_t *draws = nullptr, *Qt = nullptr;
        LaneScratch lanes;
        cudaStream_t s;
        ~Temp() {
            cudaStreamSynchronize(s);
            cudaFree(draws);
            cudaFree(Qt);
        }
    } tmp;
    tmp.s = s;
    CodeDev *const codes[2] = {&c->g, &c->g2};
    const int which[2] = {3, 4};
    const uint32_t lengths[2] = {(uint32_t)N, (uint32_t)N2};
    if ((st = sample_codes(c, *key, codes, which, lengths, &tmp.draws, s))) return fail(st);
    if ((st = tmp.lanes.alloc({{(uint32_t)N, (uint32_t)n}, {(uint32_t)N2, (uint32_t)N}}))) return fail(st);
    const size_t sw = encode_scan_status_words((uint32_t)N, (uint32_t)B);
    if (ctx_alloc(c, &c->Qs, (size_t)N * Bn) != cudaSuccess ||
        ctx_alloc(c, &c->QauxT, (size_t)N2 * N) != cudaSuccess ||
        ctx_alloc(c, &c->Yt, (size_t)m * B) != cudaSuccess ||
        ctx_alloc(c, &c->Z, (size_t)N * B) != cudaSuccess ||
        ctx_alloc(c, &c->chal2, (size_t)ell2 * 2 * t2) != cudaSuccess ||
        ctx_alloc(c, &c->R, (size_t)ell2 * Bn) != cudaSuccess ||
        ctx_alloc(c, &c->F2, (size_t)ell2 * N2) != cudaSuccess ||
        ctx_alloc(c, &c->eS, (size_t)N * B) != cudaSuccess || ctx_alloc(c, &c->estatus, sw) != cudaSuccess ||
        ctx_alloc(c, &c->status, scan_status_words((uint32_t)N2, (uint32_t)ell2)) != cudaSuccess)
        return fail(PVMVMD_E_NOMEM);
    if (cudaMemsetAsync(c->status, 0, scan_status_words((uint32_t)N2, (uint32_t)ell2) * sizeof(unsigned long long),
                        s) != cudaSuccess)
        return fail(PVMVMD_E_CUDA);
    // Q_b = G^T M_b into the column block b n of Qs (the lanes are M_b's columns)
    for (int b = 0; b < B; ++b) {
        st = encode_lanes(c->g, (uint32_t)m, (uint32_t)rate, W_dev + (size_t)b * m * n, true, (size_t)n,
                          (uint32_t)n, c->Qs + (size_t)b * n, (size_t)Bn, tmp.lanes, err, s);
        if (st) return fail(st);
    }
    // Qaux = Qt^T G': row i is G'^T applied to row i of Qs; encode with the
    // N rows of Qs as lanes, so Qs is transposed first (Qt, B n x N)
    if (dev_alloc(&tmp.Qt, (size_t)Bn * N) != cudaSuccess) return fail(PVMVMD_E_NOMEM);
    if (launch_transpose_u32(c->Qs, (int)N, (int)Bn, tmp.Qt, s) != cudaSuccess) return fail(PVMVMD_E_CUDA);
    st = encode_lanes(c->g2, Bn, (uint32_t)rate, tmp.Qt, false, (size_t)N, (uint32_t)N, c->QauxT, (size_t)N, tmp.lanes,
                      err, s);
    if (st) return fail(st);
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(PVMVMD_E_CUDA);
    if ((st = read_and_clear_error())) return fail(st);
    *out = c;
    return PVMVMD_OK;
}

int pvmvmd_bv_challenge(pvmvmd_bv_ctx *ctx, const pvmvmd_key *key, uint32_t *chal_dev, void *stream) {
    using namespace pv;
    if (!ctx || !key || !chal_dev) return PVMVMD_E_ARG;
    PV_CUDA(launch_sample_sparse(*key, kTagBvPrimary, 0, (uint32_t)ctx->N, (uint32_t)ctx->t,
                                 (uint32_t)ctx->ell, chal_dev, nullptr, 0, static_cast<cudaStream_t>(stream)));
    return PVMVMD_OK;
}

int pvmvmd_bv_server_project(const pvmvmd_bv_ctx *ctx, const uint32_t *chal_dev, uint32_t *u_dev,
                             void *stream) {
    using namespace pv;
    if (!ctx || !chal_dev || !u_dev) return PVMVMD_E_ARG;
    PV_CUDA(launch_verify_u(ctx->Qs, ctx->B * ctx->n, chal_dev, (uint32_t)ctx->t, (uint32_t)ctx->ell, u_dev,
                            static_cast<cudaStream_t>(stream)));
    return PVMVMD_OK;
}

int pvmvmd_bv_check(pvmvmd_bv_ctx *ctx, const uint32_t *X_dev, const uint32_t *Y_dev, const uint32_t *chal_dev,
                    const uint32_t *u_dev, const pvmvmd_key *key2, int32_t *accept_dev, void *stream) {
    using namespace pv;
    if (!ctx || !X_dev || !Y_dev || !chal_dev || !u_dev || !key2 || !accept_dev) return PVMVMD_E_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *err = error_word();
    if (!err) return PVMVMD_E_CUDA;
    const uint32_t Bn = (uint32_t)ctx->B * ctx->n;
    // z_b = G^T y_b (the B outputs as lanes)
    PV_CUDA(launch_transpose_u32(Y_dev, ctx->B, ctx->m, ctx->Yt, s));
    int st = encode_lanes_into(ctx->g, (uint32_t)ctx->m, (uint32_t)ctx->rate, ctx->Yt, false, (size_t)ctx->B,
                               (uint32_t)ctx->B, ctx->Z, (size_t)ctx->B, ctx->eS, ctx->estatus,
                               err, s);
    if (st) return st;
    // secondary challenges, drawn after the responses, and r^(j) = G' e'^(j)
    const CodeDev &d = ctx->g2;
    if (syndrome_tiles_eligible((uint32_t)ctx->t2)) {
        PV_CUDA(launch_syndrome_tiles(*key2, kTagBvSecondary, 0, (uint32_t)ctx->N2, (uint32_t)ctx->t2,
                                      (uint32_t)ctx->ell2, d.pi2inv, d.v2p, d.v1m, d.pi1inv, Bn,
                                      (uint32_t)ctx->rate, ctx->chal2, ctx->F2, ctx->status, err, nullptr, ctx->R,
                                      s, false));
    } else {
        PV_CUDA(launch_sample_sparse(*key2, kTagBvSecondary, 0, (uint32_t)ctx->N2, (uint32_t)ctx->t2,
                                     (uint32_t)ctx->ell2, ctx->chal2, ctx->status,
                                     scan_status_words((uint32_t)ctx->N2, (uint32_t)ctx->ell2), s));
        PV_CUDA(launch_syndrome_scan(d.pi2inv, d.v2p, d.v1, (uint32_t)ctx->N2, ctx->chal2, (uint32_t)ctx->t2,
                                     (uint32_t)ctx->ell2, ctx->F2, ctx->status, err, s));
        PV_CUDA(launch_syndrome_gather(d.pi1inv, Bn, (uint32_t)ctx->rate, ctx->F2, (uint32_t)ctx->N2, nullptr,
                                       ctx->R, (uint32_t)ctx->ell2, s));
    }
    PV_CUDA(launch_bv_checks(ctx->QauxT, ctx->N, (int)Bn, ctx->n, ctx->B, chal_dev, (uint32_t)ctx->t,
                             (uint32_t)ctx->ell, ctx->chal2, (uint32_t)ctx->t2, (uint32_t)ctx->ell2, u_dev,
                             ctx->R, X_dev, ctx->Z, accept_dev, s));
    return PVMVMD_OK;
}

int pvmvmd_bv_info(const pvmvmd_bv_ctx *ctx, pvmvmd_bv_view *v) {
    if (!ctx || !v) return PVMVMD_E_ARG;
    v->B = ctx->B; v->m = ctx->m; v->n = ctx->n; v->rate = ctx->rate; v->N = ctx->N; v->N2 = ctx->N2;
    v->t = ctx->t; v->ell = ctx->ell; v->t2 = ctx->t2; v->ell2 = ctx->ell2;
    v->Qs = ctx->Qs;
    v->QauxT = ctx->QauxT;
    v->chal2 = ctx->chal2;
    return PVMVMD_OK;
}

