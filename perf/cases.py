"""What the performance of this framework is measured on: calls of its public
entry points as a client or a server program makes them, over the sizes of the
repository's configurations (one 256 x 256 matrix up to 70B-class decoder
layers), with plain int8 or 16-bit weights, in standard and boost mode.

Every output is a whole number mod q or a verdict, so every case is exact.
"""
import math

import torch

import paper_2609_10264_gb300 as pv

Q = pv.PVMVMD_Q
RATE, T_Y, ELL = 8, 31, 2  # the paper's parameters (t_x depends on K, see _t_x)


def listed():
    return [
        # a first round trip: the smallest matrix and a single vector, where
        # launches and latency are everything
        {"name": "round_trip_256_b1", "kind": "round_trip", "m": 256, "K": 256, "B": 1, "bits": 8, "boost": False},
        # a Qwen3-4B q projection for an eight-token prompt, with 16-bit
        # weights (the paper's quantisation of FP8 models)
        {"name": "round_trip_4096x2560_b8_i16", "kind": "round_trip", "m": 4096, "K": 2560, "B": 8, "bits": 16,
         "boost": False},
        # sizes that no tile divides, in boost mode (masks made ahead while
        # the client was idle): add the masks, multiply, verify and unmask
        {"name": "boost_1030x1001_b70", "kind": "round_trip", "m": 1030, "K": 1001, "B": 70, "bits": 8, "boost": True},
        # the server's work for one token through eight 8B-class layers: four
        # dependent calls a layer, each product with its own masked vector
        {"name": "server_token_8b", "kind": "token", "hidden": 4096, "kv": 1024, "ffn": 14336, "layers": 8},
        # a server with a hundred independent requests at hand, one vector each
        {"name": "server_4096_100_requests", "kind": "requests", "m": 4096, "K": 4096, "count": 100, "copies": 64},
        # the server's work for one 8B-class layer and a batch of 64 vectors
        {"name": "server_layer_8b_b64", "kind": "layer", "hidden": 4096, "kv": 1024, "ffn": 14336, "B": 64},
        # the largest: one 70B-class layer and a batch of 256 vectors
        {"name": "server_layer_70b_b256", "kind": "layer", "hidden": 8192, "kv": 1024, "ffn": 28672, "B": 256},
        # the client masks a batch: a code that fits one SM, and a longer one
        {"name": "encode_4096_b100", "kind": "encode", "m": 1024, "K": 4096, "B": 100},
        {"name": "encode_8192_b256", "kind": "encode", "m": 1024, "K": 8192, "B": 256},
        # the client verifies and unmasks a batch of answers
        {"name": "decode_4096_b100", "kind": "decode", "m": 4096, "K": 4096, "B": 100},
        {"name": "decode_14336x4096_b64", "kind": "decode", "m": 14336, "K": 4096, "B": 64},
        # the client prepares for one matrix (once per matrix: a model has hundreds)
        {"name": "preprocess_4096", "kind": "preprocess", "m": 4096, "K": 4096},
    ]


def _log(rng, lo, hi, step=1):
    """A size spread over the logarithm of [lo, hi], a multiple of step."""
    v = int(round(lo * (hi / lo) ** rng.random()))
    return max(step, min(hi, v // step * step))


def draw(rng):
    kind = rng.choice(["round_trip", "round_trip", "boost", "token", "requests", "layer", "encode", "decode",
                       "preprocess"])
    # projections are mostly multiples of 16 wide; any other width is taken too
    step = rng.choice([1, 16, 16, 64])
    if kind in ("round_trip", "boost"):
        return {"kind": "round_trip", "m": _log(rng, 32, 4096), "K": _log(rng, 32, 4096, step),
                "B": _log(rng, 1, 96), "bits": rng.choice([8, 8, 16]), "boost": kind == "boost"}
    if kind == "token":
        hidden = _log(rng, 512, 4096, step)
        return {"kind": kind, "hidden": hidden, "kv": max(16, hidden // rng.choice([1, 2, 4, 8]) // 16 * 16),
                "ffn": _log(rng, 2 * hidden, 7 * hidden // 2, step), "layers": rng.randint(1, 8)}
    if kind == "requests":
        return {"kind": kind, "m": _log(rng, 128, 4096), "K": _log(rng, 128, 4096, step),
                "count": _log(rng, 2, 100), "copies": rng.choice([1, 16, 64])}
    if kind == "layer":
        hidden = _log(rng, 512, 6144, 16)
        return {"kind": kind, "hidden": hidden, "kv": max(64, hidden // rng.choice([1, 4, 8]) // 16 * 16),
                "ffn": _log(rng, 2 * hidden, 7 * hidden // 2, 16), "B": _log(rng, 2, 256)}
    if kind == "encode":
        K = _log(rng, 256, 16384, step)
        return {"kind": kind, "m": _log(rng, 64, 1024), "K": K, "B": _log(rng, 1, min(256, (8192 * 256) // K))}
    if kind == "decode":
        m = _log(rng, 256, 14336)
        return {"kind": kind, "m": m, "K": _log(rng, 256, 4096, step), "B": _log(rng, 1, min(256, (14336 * 64) // m))}
    return {"kind": kind, "m": _log(rng, 64, 4096), "K": _log(rng, 64, 4096, step)}


# ---------------------------------------------------------------- inputs

class _Random:
    """Tensors on the GPU from a seed alone."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def _normal(self, m, K, sigma, limit, dtype):
        out = torch.empty((m, K), dtype=dtype, device="cuda")
        for r in range(0, m, 4096):  # in blocks of rows, to bound the float copy
            g = torch.randn((min(4096, m - r), K), generator=self.g, device="cuda")
            out[r:r + 4096] = (g * sigma).round_().clamp_(-limit, limit).to(dtype)
        return out

    def weights(self, m, K):
        """Quantised weights: a Gaussian, rounded and clipped."""
        return self._normal(m, K, 32.0, 127, torch.int8)

    def weights16(self, m, K):
        return self._normal(m, K, 2048.0, 32000, torch.int16)

    def plain(self, B, K):
        """Quantised activations in [-127, 127]."""
        return torch.randint(-127, 128, (B, K), generator=self.g, device="cuda", dtype=torch.int64)

    def field(self, B, K):
        """Masked vectors: uniform in F_q."""
        return torch.randint(0, Q, (B, K), generator=self.g, device="cuda", dtype=torch.int64).to(torch.int32)

    def key(self):
        w = torch.randint(0, 1 << 32, (8,), generator=self.g, device="cuda", dtype=torch.int64)
        return [int(v) for v in w.cpu()]


def _embed(x):
    """Signed integers -> F_q, as 32-bit words."""
    return (x % Q).to(torch.int32)


def _i32(*shape):
    return torch.empty(shape, dtype=torch.int32, device="cuda")


def _projections(case):
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    return [[(h, h), (kv, h), (kv, h)], [(h, h)], [(f, h), (f, h)], [(h, f)]]  # q k v, o, gate up, down


def _make(case, seed):
    """The tensors of a case, from its seed: (random source, weights, vectors)."""
    r = _Random(seed)
    kind = case["kind"]
    if kind in ("round_trip", "encode", "decode", "preprocess"):
        m, K = case["m"], case["K"]
        W = r.weights16(m, K) if case.get("bits") == 16 else r.weights(m, K)
        return r, W, None if kind == "preprocess" else r.plain(case["B"], K)
    if kind == "requests":
        n, m, K = case["count"], case["m"], case["K"]
        return r, [r.weights(m, K) for _ in range(min(case["copies"], n))], r.field(n, K)
    shapes = [s for call in _projections(case) for s in call]
    if kind == "layer":
        return r, [r.weights(*s) for s in shapes], [r.field(case["B"], K) for _, K in shapes]
    n = case["layers"]
    return r, [r.weights(*s) for _ in range(n) for s in shapes], [r.field(1, K)[0] for _ in range(n) for _, K in shapes]


def prepare(case, seed):
    kind = case["kind"]
    r, W, X = _make(case, seed)
    s = {"kind": kind, "W": W, "X": X}
    if kind == "requests":
        s["Y"] = _i32(case["count"], case["m"])
        s["jobs"] = pv.mvm_jobs([(W[i % len(W)], X[i], s["Y"][i]) for i in range(case["count"])])
    elif kind == "layer":
        s["Y"] = [_i32(case["B"], w.shape[0]) for w in W]
        s["jobs"] = pv.batch_jobs(list(zip(W, X, s["Y"])))
    elif kind == "token":
        s["Y"] = [_i32(w.shape[0]) for w in W]
        s["calls"], at = [], 0
        for _ in range(case["layers"]):
            for call in _projections(case):
                part = slice(at, at + len(call))
                s["calls"].append(pv.mvm_jobs(list(zip(W[part], X[part], s["Y"][part]))))
                at += len(call)
    else:
        s["keys"] = [pv.make_key(r.key()) for _ in range(3)]
        if kind == "preprocess":
            return s
        B, m, K = case["B"], case["m"], case["K"]
        wide = case.get("bits") == 16
        params = pv.pvmvmd_params()
        params.scratch_batch = B  # a batch is one encode
        ctx = s["ctx"] = (pv.pvmvmd_preprocess_i16 if wide else pv.pvmvmd_preprocess)(W, s["keys"][0], params)
        s["X"], s["Xh"], s["st"] = _embed(X), _i32(B, K), _i32(B, 2 * ctx.t_x)
        s["Yh"], s["Y"], s["ok"] = _i32(B, m), _i32(B, m), _i32(B)
        if kind == "round_trip":
            s["planes"] = pv.pvmvmd_weights_split_i16(W) if wide else None
            s["tmp"] = _i32(B, m) if wide else None
            s["masks"] = pv.pvmvmd_boost_prepare(ctx, B, s["keys"][1]) if case["boost"] else None
        elif kind == "decode":
            pv.pvmvmd_encode(ctx, s["X"], s["keys"][1], s["Xh"], s["st"])
            pv.pvmvmd_server_mvm(W, s["Xh"], s["Yh"])
            # the last of several answers is a wrong one, which the client rejects
            if B > 1:
                s["Yh"][-1, m // 2] = (s["Yh"][-1, m // 2].to(torch.int64) + 1) % Q
    return s


def run(s):
    kind = s["kind"]
    if kind == "requests":
        pv.pvmvmd_server_mvm_multi(s["jobs"])
        return s["Y"]
    if kind == "layer":
        pv.pvmvmd_server_mvm_grouped(s["jobs"])
        return s["Y"]
    if kind == "token":
        for jobs in s["calls"]:
            pv.pvmvmd_server_mvm_multi(jobs)
        return s["Y"]
    if kind == "preprocess":
        ctx = pv.pvmvmd_preprocess(s["W"], s["keys"][0])
        v = pv.pvmvmd_ctx_info(ctx)
        out = [pv.device_view(v.PT, v.N_x * v.m).view(v.N_x, v.m), pv.device_view(v.Q, v.N_y * v.K).view(v.N_y, v.K)]
        for t in out:
            t.ctx = ctx  # the context owns the memory: it lives as long as either output does
        return out
    ctx, keys = s["ctx"], s["keys"]
    if kind == "encode":
        pv.pvmvmd_encode(ctx, s["X"], keys[1], s["Xh"], s["st"])
        return [s["Xh"], s["st"]]
    if kind == "decode":
        pv.pvmvmd_decode_verify(ctx, s["st"], s["Xh"], s["Yh"], keys[2], s["Y"], s["ok"])
        return [s["Y"], s["ok"]]
    masks, planes = s["masks"], s["planes"]
    if masks:
        pv.pvmvmd_boost_encode(s["X"], masks[0], s["Xh"])
    else:
        pv.pvmvmd_encode(ctx, s["X"], keys[1], s["Xh"], s["st"])
    if planes:
        pv.pvmvmd_server_mvm_i16(planes[0], planes[1], s["Xh"], s["Yh"], s["tmp"])
    else:
        pv.pvmvmd_server_mvm(s["W"], s["Xh"], s["Yh"])
    if masks:
        pv.pvmvmd_boost_decode_verify(ctx, masks[1], s["Xh"], s["Yh"], keys[2], s["Y"], s["ok"])
    else:
        pv.pvmvmd_decode_verify(ctx, s["st"], s["Xh"], s["Yh"], keys[2], s["Y"], s["ok"])
    return [s["Xh"], s["Yh"], s["Y"], s["ok"]]


# ---------------------------------------------------------------- work

def _t_x(K):
    """The mask's sparsity, Eq. (1): ceil(ln 2 (128 - log2 N_x) / delta), delta = 1/2."""
    return math.ceil(2 * math.log(2.0) * (128 - math.log2(RATE * K)))


def work(case):
    """Bytes read and written once, and two operations for a multiply-add in
    F_q.  A mask costs the four operations per position of its code (a sum, a
    scaling, twice), an unmasking t_x multiply-adds per output; verification
    reads t_y rows of Q per challenge and takes a product per entry."""
    kind = case["kind"]

    def product(m, K, B, bits=8):
        return m * K * bits // 8 + 4 * B * (m + K), 2 * m * K * B * bits // 8

    def encode(K, B):
        return 4 * (B * (2 * K + 2 * _t_x(K)) + 4 * RATE * K), 4 * RATE * K * B

    def unmask(m, K, B):
        # at most N_x distinct rows of P^T for the batch
        rows = min(B * _t_x(K), RATE * K)
        return 4 * (rows * m + 2 * B * m + 2 * B * _t_x(K)), 2 * B * _t_x(K) * m

    def verify(m, K, B):
        return (4 * (ELL * T_Y * K + 4 * RATE * m + B * (K + m) + B),
                ELL * (2 * T_Y * K + 4 * RATE * m + 2 * B * (K + m)))

    if kind == "requests":
        parts = [product(case["m"], case["K"], 1)] * case["count"]
    elif kind in ("layer", "token"):
        shapes = [s for call in _projections(case) for s in call]
        parts = [product(m, K, case.get("B", 1)) for m, K in shapes] * case.get("layers", 1)
    elif kind == "preprocess":
        m, K = case["m"], case["K"]
        parts = [(m * K + 2 * 4 * RATE * m * K, 2 * 4 * RATE * m * K)]
    else:
        m, K, B = case["m"], case["K"], case["B"]
        if kind == "encode":
            parts = [encode(K, B)]
        elif kind == "decode":
            parts = [unmask(m, K, B), verify(m, K, B)]
        elif case["boost"]:
            parts = [(12 * B * K, B * K), product(m, K, B, case["bits"]), (12 * B * m, B * m), verify(m, K, B)]
        else:
            parts = [encode(K, B), product(m, K, B, case["bits"]), unmask(m, K, B), verify(m, K, B)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------- the same by plain arithmetic

def _times(W, X):
    """X W^T mod q for X in [0, q) (B x K): the two 16-bit halves of X by 64-bit
    float products, exact since |W| 2^16 K < 2^53."""
    y = 0
    for shift in (16, 0):
        half = ((X.to(torch.int64) >> shift) & 0xFFFF).to(torch.float64)
        part = torch.cat([half @ W[r:r + 4096].to(torch.float64).T for r in range(0, W.shape[0], 4096)], 1)
        y = (y * 65536 + part.to(torch.int64)) % Q
    return y


def exact(case, seed):
    """What does not rest on the random masks and codes: the products, the
    unmasked results and the verdicts."""
    kind = case["kind"]
    if kind in ("encode", "preprocess"):
        return None
    _, W, X = _make(case, seed)
    if kind == "requests":
        return torch.cat([_times(W[i % len(W)], X[i:i + 1]) for i in range(case["count"])]).to(torch.int32)
    if kind == "layer":
        return [_times(w, x).to(torch.int32) for w, x in zip(W, X)]
    if kind == "token":
        return [_times(w, x[None])[0].to(torch.int32) for w, x in zip(W, X)]
    Y = _times(W, X % Q)
    ok = torch.ones(case["B"], dtype=torch.int32, device="cuda")
    if kind == "decode":
        if case["B"] > 1:
            Y[-1, case["m"] // 2] = (Y[-1, case["m"] // 2] + 1) % Q
            ok[-1] = 0
        return [Y.to(torch.int32), ok]
    return [None, None, Y.to(torch.int32), ok]
