"""What the framework's users run, as measurable cases.

Every case goes through `paper_2505_14638_b200.binding`, with the buffers, prepacked weights and
workspaces that a serving engine (or a calibration script) keeps.  The kinds:

  layer      one linear layer: per-token activation quantization, then the W4A8 matrix product
  block      the four linears of a decoder block in sequence, one call per step, each with the
             quantization of its own input (what lies between them is the engine's)
  chain      a list of independent decode-sized layers in one launch
  chain_mlp  the gated MLP of a decoder block as a dependent chain in one launch
  hessian    calibration: X^T X of two batches of calibration tokens
  dpq        the weight quantizer on one layer (order, scale search, asymmetric or symmetric)

Weights are drawn from N(0, sigma^2) and quantized with the framework's round-to-nearest quantizer;
activations are BF16 N(0, 1) with one channel in a hundred scaled by 20.
"""
import math

import torch

from paper_2505_14638_b200 import binding

MAX_FLOPS = 2.0 * 8192 * 8192 * 28672      # the largest prefill layer: no drawn product exceeds it
MAX_DPQ = 4096 * 14336 * 14336             # N K^2 of the largest quantized layer


def listed():
    return [
        # the smallest layer of the benchmark's configurations: latency and launches
        dict(name="layer_small_m16", kind="layer", M=16, K=1024, N=1024, weights="signmag", per_channel=False,
             out="bf16", scale="exact"),
        # the benchmark's decode sweep: eight steps of M = 1, 4, 16 on the up-projection shape
        dict(name="decode_sweep", kind="chain", count=24, M0=1, M1=4, M2=16, K=4096, N=14336, weights="signmag"),
        # decoding one token for a few sequences: an asymmetric MLP as a dependent chain
        dict(name="decode_mlp_asym", kind="chain_mlp", M=4, hidden=4096, ffn=14336, weights="tiled"),
        # decoding with one call per layer, as an engine that has other work between the layers
        dict(name="block_decode_m8", kind="block", M=8, hidden=4096, kv=1024, ffn=14336, weights="signmag",
             per_channel=False),
        # a ragged batch of sequences (continuous batching), asymmetric weights, per-channel weight scale
        dict(name="block_batch_m77", kind="block", M=77, hidden=4096, kv=1024, ffn=14336, weights="tiled",
             per_channel=True),
        # a short prompt, or a large decode batch
        dict(name="block_m512", kind="block", M=512, hidden=4096, kv=1024, ffn=14336, weights="signmag",
             per_channel=False),
        # prefill of the attention output projection
        dict(name="prefill_o_m2048", kind="layer", M=2048, K=4096, N=4096, weights="signmag", per_channel=False,
             out="bf16", scale="exact"),
        # prefill of a ragged prompt through a whole block, asymmetric weights
        dict(name="block_prefill_m1531", kind="block", M=1531, hidden=4096, kv=1024, ffn=14336, weights="tiled",
             per_channel=True),
        # the largest prefill layer
        dict(name="prefill_large", kind="layer", M=8192, K=8192, N=28672, weights="signmag", per_channel=False,
             out="bf16", scale="exact"),
        # weights in the boundary format (no prepacking), FP32 result, power-of-two activation scales
        dict(name="canonical_m33_fp32", kind="layer", M=33, K=4096, N=6144, weights="canonical", per_channel=True,
             out="fp32", scale="pow2"),
        # calibration of a layer: two batches of tokens
        dict(name="hessian_k4096", kind="hessian", T=2048, K=4096),
        # quantizing the largest reduction of a block: the down projection
        dict(name="dpq_down", kind="dpq", N=4096, K=14336, symmetric=False, mse_steps=6),
    ]


def _log_int(rng, lo, hi, mult=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / mult)) * mult))


def draw(rng):
    while True:
        kind = rng.choice(["layer", "layer", "block", "block", "chain", "chain_mlp", "hessian", "dpq"])
        weights = rng.choice(["signmag", "tiled"])
        if kind == "layer":
            case = dict(kind=kind, M=_log_int(rng, 1, 8192), K=_log_int(rng, 1024, 14336, 128),
                        N=_log_int(rng, 1024, 28672, 16), weights=rng.choice(["signmag", "tiled", "canonical"]),
                        per_channel=rng.random() < 0.5, out=rng.choice(["bf16", "bf16", "fp32"]),
                        scale=rng.choice(["exact", "exact", "pow2"]))
        elif kind == "block":
            hidden = _log_int(rng, 1024, 8192, 128)
            case = dict(kind=kind, M=_log_int(rng, 1, 4096), hidden=hidden,
                        kv=rng.choice([hidden // 4, hidden // 8]) // 16 * 16,
                        ffn=min(14336, int(hidden * rng.uniform(2.5, 3.6)) // 128 * 128), weights=weights,
                        per_channel=rng.random() < 0.5)
        elif kind == "chain":
            case = dict(kind=kind, count=rng.randint(1, 24), M0=rng.randint(1, 16), M1=rng.randint(1, 16),
                        M2=rng.randint(1, 16), K=_log_int(rng, 1024, 8192, 128), N=_log_int(rng, 1024, 14336, 16),
                        weights=weights)
        elif kind == "chain_mlp":
            hidden = _log_int(rng, 1024, 8192, 128)
            case = dict(kind=kind, M=rng.randint(1, 16), hidden=hidden,
                        ffn=min(14336, int(hidden * rng.uniform(2.5, 3.6)) // 128 * 128), weights=weights)
        elif kind == "hessian":
            case = dict(kind=kind, T=_log_int(rng, 256, 4096), K=_log_int(rng, 1024, 8192, 128))
        else:
            case = dict(kind=kind, N=_log_int(rng, 256, 8192, 16), K=_log_int(rng, 1024, 8192, 128),
                        symmetric=rng.random() < 0.5, mse_steps=rng.choice([0, 6, 11]))
            if case["N"] * case["K"] ** 2 > MAX_DPQ:
                continue
        if work(case)["flops"] <= MAX_FLOPS:
            return case


# ---- preparation ---------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _activation(g, M, K):
    x = torch.randn((M, K), generator=g, device="cuda")
    cols = torch.randperm(K, generator=g, device="cuda")[:max(1, K // 100)]
    x[:, cols] *= 20.0
    return x.to(torch.bfloat16)


class _Layer:
    """A quantized layer with the buffers a serving engine keeps for it."""

    def __init__(self, g, M, N, K, weights, per_channel, out="bf16"):
        W = torch.randn((N, K), generator=g, device="cuda") * 0.02
        codes, gscale, gzero, s_w = binding.quantize_weight_rtn(W, symmetric=weights == "signmag",
                                                                per_channel=per_channel)
        if weights == "canonical":
            self.w = (codes, gscale, gzero, s_w)
        else:
            self.w = binding.prepack_weight(codes, gscale, gzero, s_w)
        self.canonical = weights == "canonical"
        self.out_dtype = binding.OUT_FP32 if out == "fp32" else binding.OUT_BF16
        self.y = torch.empty((M, N), dtype=torch.float32 if out == "fp32" else torch.bfloat16, device="cuda")
        self.x8 = torch.empty((M, K), dtype=torch.uint8, device="cuda")
        self.s_x = torch.empty((M,), dtype=torch.float32, device="cuda")
        fmt = binding.FMT_CANONICAL if self.canonical else self.w.fmt
        self.ws = binding.new_workspace(M, N, K, fmt)

    def __call__(self, x, scale_mode=binding.SCALE_EXACT):
        binding.quantize_act(x, scale_mode=scale_mode, out=(self.x8, self.s_x))
        if self.canonical:
            return binding.linear(self.x8, self.s_x, *self.w, out_dtype=self.out_dtype, out=self.y, workspace=self.ws)
        return binding.linear_tiled(self.x8, self.s_x, self.w, out_dtype=self.out_dtype, out=self.y, workspace=self.ws)


def _block_shapes(c):
    h, f = c["hidden"], c["ffn"]
    return (("qkv", h + 2 * c["kv"], h), ("o", h, h), ("gate_up", 2 * f, h), ("down", h, f))


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    st = dict(case=case)
    if kind == "layer":
        st["x"] = _activation(g, case["M"], case["K"])
        st["layer"] = _Layer(g, case["M"], case["N"], case["K"], case["weights"], case["per_channel"], case["out"])
        st["mode"] = binding.SCALE_POW2 if case["scale"] == "pow2" else binding.SCALE_EXACT
    elif kind == "block":
        M = case["M"]
        st["layers"] = [(name, _activation(g, M, K), _Layer(g, M, N, K, case["weights"], case["per_channel"]))
                        for name, N, K in _block_shapes(case)]
    elif kind in ("chain", "chain_mlp"):
        if kind == "chain":
            shapes = [((case["M0"], case["M1"], case["M2"])[i % 3], case["N"], case["K"]) for i in range(case["count"])]
        else:
            shapes = [(case["M"], 2 * case["ffn"], case["hidden"]), (case["M"], case["hidden"], case["ffn"])]
        problems = []
        for i, (M, N, K) in enumerate(shapes):
            lay = _Layer(g, M, N, K, case["weights"], False)
            if kind == "chain_mlp" and i == 1:
                p = dict(x=problems[0]["y"], weight=lay.w, y=lay.y, kind=binding.CHAIN_INPUT_SILU_MUL, depends_on=0)
            else:
                p = dict(x=_activation(g, M, K), weight=lay.w, y=lay.y)
            problems.append(p)
        st["chain"] = binding.LinearChain(problems)
        st["y"] = [p["y"] for p in problems]
    elif kind == "hessian":
        st["batches"] = _activation(g, case["T"], case["K"]).chunk(2)
    else:
        N, K = case["N"], case["K"]
        st["W"] = torch.randn((N, K), generator=g, device="cuda") * 0.02
        # correlated calibration features of uneven strength, then the caller's library factorization
        X = _activation(g, 2048, K).float() + 0.5 * torch.randn((2048, 1), generator=g, device="cuda")
        X = (X * torch.linspace(0.3, 3.0, K, device="cuda")[torch.randperm(K, generator=g, device="cuda")]).bfloat16()
        H = binding.hessian_accumulate(X)
        del X
        st["perm"] = binding.gar_permutation(H.diagonal().contiguous())
        Hp = binding.hessian_prepare(H, st["perm"]).to(torch.float64)
        del H
        Hinv = torch.cholesky_inverse(torch.linalg.cholesky(Hp))
        del Hp
        Hinv = 0.5 * (Hinv + Hinv.T)
        st["U"] = torch.linalg.cholesky(Hinv, upper=True).to(torch.float32).contiguous()
    return st


# ---- one pass ------------------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "layer":
        return st["layer"](st["x"], st["mode"])
    if kind == "block":
        return {name: layer(x) for name, x, layer in st["layers"]}
    if kind in ("chain", "chain_mlp"):
        st["chain"]()
        return st["y"]
    if kind == "hessian":
        H = None
        for x in st["batches"]:
            H = binding.hessian_accumulate(x, H)
        return H
    codes, gscale, gzero, s_w = binding.dpq_quantize(st["W"], st["U"], st["perm"], symmetric=case["symmetric"],
                                                     mse_steps=case["mse_steps"])
    out = dict(codes=codes, gscale=gscale, s_w=s_w)
    if gzero is not None:
        out["gzero"] = gzero
    return out


# ---- what a pass cannot do without -----------------------------------------------------------------
def _linear_work(M, N, K, symmetric, per_channel=False, out_bytes=2, x_bytes=2):
    weights = N * K // 2 + (2 if symmetric else 3) * N * (K // 128) + 4 * (N if per_channel else 1)
    return weights + x_bytes * M * K + out_bytes * M * N, 2.0 * M * N * K


def work(case):
    kind = case["kind"]
    sym = case.get("weights") == "signmag"
    if kind == "layer":
        parts = [_linear_work(case["M"], case["N"], case["K"], sym, case["per_channel"], 4 if case["out"] == "fp32" else 2)]
    elif kind == "block":
        parts = [_linear_work(case["M"], N, K, sym, case["per_channel"]) for name, N, K in _block_shapes(case)]
    elif kind == "chain":
        parts = [_linear_work((case["M0"], case["M1"], case["M2"])[i % 3], case["N"], case["K"], sym)
                 for i in range(case["count"])]
    elif kind == "chain_mlp":
        parts = [_linear_work(case["M"], 2 * case["ffn"], case["hidden"], sym),
                 _linear_work(case["M"], case["hidden"], case["ffn"], sym, x_bytes=4)]
    elif kind == "hessian":
        T, K = case["T"], case["K"]
        parts = [(2 * T * K + 4 * K * K, 1.0 * T * K * (K + 1))]   # one triangle of X^T X
    else:
        N, K = case["N"], case["K"]
        parts = [(4 * N * K + 2 * K * (K + 1) + 4 * K + N * K // 2 + (2 if case["symmetric"] else 3) * N * (K // 128),
                  1.0 * N * K * (K - 1))]                           # Eq. 12: one FMA per weight and later column
    return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))


# ---- how far another correct implementation may be ------------------------------------------------
def tolerance(case):
    # Measured against the same FP8 operands multiplied in float64 (the hessian: X^T X in float64) over the
    # listed and some drawn cases; about four times the largest difference seen.
    kind = case["kind"]
    if kind == "dpq":
        return "exact"                      # integer codes; every deciding step is one fp32 operation
    if kind == "hessian":
        return {"rel": 1e-5, "max": 4e-5}   # seen 2.2e-6 / 6.1e-6
    if kind == "chain_mlp":
        return {"rel": 1.6e-3, "max": 0.03}   # seen 4.0e-4 / 7.8e-3: a BF16 step before the second quantization
    if kind == "layer" and case["out"] == "fp32":
        return {"rel": 1e-6, "max": 1e-5}   # seen 8.6e-8 / 4.0e-7 at K <= 4736; grows with K
    return {"rel": 1.6e-4, "max": 0.016}    # seen 4.7e-5 / 7.8e-3: one BF16 step where the FP32 sums round apart


# ---- the same in 64 bits ---------------------------------------------------------------------------
# Every FP8 operand, code and scale is decided by single FP32 operations that torch performs alike;
# the products, sums and output scales below are float64, the outputs unrounded.
def _e4m3(v):
    return v.clamp(-448.0, 448.0).to(torch.float8_e4m3fn).to(torch.float32)


def _pow2_ceil(s):
    m, e = torch.frexp(s)
    return torch.where(m == 0.5, s, torch.ldexp(torch.ones_like(s), e))


def _exact_weight(g, N, K, weights, per_channel):
    """The float64 weights that inference multiplies with: FP8 values times their weight scale."""
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    amax = W.abs().amax(dim=1, keepdim=True) if per_channel else W.abs().max().reshape(1, 1)
    s_w = amax / torch.full_like(amax, 448.0)
    w8 = _e4m3(W / s_w).view(N, K // 128, 128)
    del W
    if weights == "signmag":
        a = w8.abs().amax(dim=2, keepdim=True)
        s = (a / torch.full_like(a, 7.0)).bfloat16().float()
        q = (w8 / s).round().clamp(-7.0, 7.0)
    else:
        lo, hi = w8.amin(dim=2, keepdim=True).clamp(max=0.0), w8.amax(dim=2, keepdim=True).clamp(min=0.0)
        s = ((hi - lo) / torch.full_like(hi, 15.0)).bfloat16().float()
        z = (-lo / s).round().clamp(0.0, 15.0)
        q = (w8 / s + z).round().clamp(0.0, 15.0) - z
    return _e4m3(q * s).view(N, K).double() * s_w.double()


def _exact_linear(x, w, scale="exact"):
    x = x.float()
    amax = x.abs().amax(dim=1, keepdim=True)
    top = torch.full_like(amax, 448.0)
    s = amax / top
    inv = top / amax
    if scale == "pow2":
        s = _pow2_ceil(s)
        inv = torch.ones_like(s) / s
    return (_e4m3(x * inv).double() @ w.T).mul_(s.double())


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "layer":
        x = _activation(g, case["M"], case["K"])
        return _exact_linear(x, _exact_weight(g, case["N"], case["K"], case["weights"], case["per_channel"]),
                             case["scale"])
    if kind == "block":
        out = {}
        for name, N, K in _block_shapes(case):
            x = _activation(g, case["M"], K)
            out[name] = _exact_linear(x, _exact_weight(g, N, K, case["weights"], case["per_channel"]))
        return out
    if kind == "chain":
        out = []
        for i in range(case["count"]):
            M = (case["M0"], case["M1"], case["M2"])[i % 3]
            w = _exact_weight(g, case["N"], case["K"], case["weights"], False)
            out.append(_exact_linear(_activation(g, M, case["K"]), w))
        return out
    if kind == "chain_mlp":
        M, h, f = case["M"], case["hidden"], case["ffn"]
        w = _exact_weight(g, 2 * f, h, case["weights"], False)
        gate_up = _exact_linear(_activation(g, M, h), w)
        w = _exact_weight(g, h, f, case["weights"], False)
        stored = gate_up.bfloat16().double()          # what the second layer reads is BF16 by definition
        act = (stored[:, :f] * torch.sigmoid(stored[:, :f]) * stored[:, f:]).bfloat16()
        return [gate_up, _exact_linear(act, w)]
    if kind == "hessian":
        x = _activation(g, case["T"], case["K"]).double()
        return x.T @ x
    return None                                       # the quantizer: whole numbers
