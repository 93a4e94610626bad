"""Performance cases of the fused quantized linear layer: what its users run, over the range of sizes they run it at.

A case is one pass of a program that holds calibrated layers on the GPU: the linears of one transformer block back to
back, or a single linear, in one of the four main formats (`main`) with one of the branch formats (`branch`) and a rank,
through one of the public entry points (`entry`):
  device   lq_quantize_act + lq_linear_forward, X and Y in GPU memory
  static   lq_linear_forward_static, the call for programs that may not allocate (SINT4 layers, small M)
  host     lq_linear_forward_host, X and Y in pinned host memory
`shapes` lists the linears as "KxN" (K input features, N output features), `M` the rows (tokens x batch), `out` the
output type, `bias` whether the layers carry one.
"""
import math

import torch

from paper_2604_18117_b200 import binding as B
from paper_2604_18117_b200.inputs import PIXART_LAYERS, SANA_LAYERS

PIXART = ",".join(f"{s.K}x{s.N}" for s in PIXART_LAYERS)
SANA = ",".join(f"{s.K}x{s.N}" for s in SANA_LAYERS)


def _case(name, shapes, M, main="sint4", branch="w8a8", rank=32, entry="device", out="f16", bias=False):
    return {"name": name, "entry": entry, "main": main, "branch": branch, "rank": rank, "M": M, "shapes": shapes,
            "out": out, "bias": bias}


def listed():
    return [
        # one conditioning vector (a timestep embedding's projection): launches and latency are all there is
        _case("row", "1152x1152", 1, bias=True),
        # a short caption through an MLP's first linear, in a server that may not allocate
        _case("static-120", "1152x4608", 120, entry="static", out="f32", bias=True),
        # the smallest configuration of the benchmark: 256 tokens
        _case("tokens-256", "1152x1152", 256, main="mxint4"),
        # no size a multiple of a tile, full-precision branch, fp32 output
        _case("ragged-1365", "1160x2312,2312x1160", 1365, main="mxint4", branch="w16a16", rank=24, out="f32", bias=True),
        # the benchmark's block: 4096 tokens x batch 2 through a PixArt-class block's four linears, in each main format
        _case("block-sint4", PIXART, 8192),
        _case("block-mxint4", PIXART, 8192, main="mxint4"),
        _case("block-mxfp4", PIXART, 8192, main="mxfp4", branch="mxfp8", rank=64),
        _case("block-mxint4a8", PIXART, 8192, main="mxint4a8", branch="mxint8", rank=64),
        # the SANA-class block (N not a multiple of 128, K of 5600), biased, with the widest factors and the narrowest
        _case("wide-mxfp4", SANA, 8192, main="mxfp4", branch="mxfp4", rank=128, bias=True),
        _case("wide-sint4", SANA, 8192, branch="w4a8", bias=True),
        # the largest batch of the benchmark: 8 x 4096 tokens through one block of the stack
        _case("stack-32768", PIXART, 32768),
        # an application whose activations live in host memory
        _case("host-4096", "1152x1152", 4096, main="mxint4", entry="host"),
    ]


# (main, branch, largest rank)
_FORMATS = [("sint4", "w8a8", 128), ("sint4", "w6a6", 128), ("sint4", "w4a8", 128), ("sint4", "w16a16", 64),
            ("mxint4", "w8a8", 128), ("mxint4", "w4a8", 128), ("mxint4", "w16a16", 64),
            ("mxfp4", "mxfp8", 64), ("mxfp4", "mxfp6", 86), ("mxfp4", "mxfp4", 128),
            ("mxint4a8", "mxint8", 64), ("mxint4a8", "mxint4", 128), ("sint4", "none", 0), ("mxint4", "none", 0)]
_LARGEST = 32768 * sum(s.K * s.N for s in PIXART_LAYERS)


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One linear of any size the layers take: M over 1 .. 32768, K and N over 256 .. 8192 in steps of 8."""
    entry = rng.choice(["device"] * 6 + ["static", "host"])
    main, branch, top = rng.choice([f for f in _FORMATS if entry != "static" or f[0] == "sint4"])
    K, N = (8 * round(_spread(rng, 256, 8192) / 8) for _ in range(2))
    M = round(_spread(rng, 1, 256 if entry == "static" else 8192 if entry == "host" else 32768))
    M = max(1, min(M, _LARGEST // (K * N)))
    rank = 0 if top == 0 else min(top, rng.choice([16, 24, 32, 32, 48, 64, 86, 128]))
    c = _case("", f"{K}x{N}", M, main, branch, rank, entry, rng.choice(["f16", "f16", "f32"]), rng.random() < 0.5)
    del c["name"]
    return c


# ---- quantized layers, as lq_layer_import takes them ------------------------------------------------------------------
def _rows(v, n):
    """[G, cols] -> [G * n, cols]: each block's scale under every row of the block."""
    return v.repeat_interleave(n, 0)


def _block_max(v, n):
    """Largest magnitude of each block of n along axis 0 (the last one may be short) and of each column."""
    pad = -v.shape[0] % n
    return torch.nn.functional.pad(v.abs(), (0, 0, 0, pad)).reshape(-1, n, v.shape[1]).amax(1)


def _pow2_scale(a, qmax, lo=-24, hi=15):
    """The smallest power of two that does not clip: qmax 2^e >= a."""
    return torch.exp2(torch.log2(a.clamp_min(2.0 ** -120) / qmax).ceil().clamp(lo, hi))


_GRID = {"mxfp4": [0, .5, 1, 1.5, 2, 3, 4, 6], "mxfp6": [m / 8 for m in range(8)] + [(8 + m) / 8 * 2 ** e for e in range(3) for m in range(8)]}
_EMAX = {"mxfp8": 8, "mxfp6": 2, "mxfp4": 2}


def _mxfp(v, fmt):
    """Block-of-32 MXFP elements along axis 0: (element values, scales 2^e)."""
    s = torch.exp2(torch.log2(_block_max(v, 32).clamp_min(2.0 ** -20)).floor() - _EMAX[fmt])
    x = v / _rows(s, 32)[: v.shape[0]]
    if fmt == "mxfp8":
        return x.clamp(-448, 448).to(torch.float8_e4m3fn).float(), s
    grid = torch.tensor(_GRID[fmt], device=v.device)
    at = torch.bucketize(x.abs().contiguous(), (grid[1:] + grid[:-1]) / 2)
    return grid[at] * x.sign(), s


def _ints(v, qmax, n):
    """MX integer codes in blocks of n along axis 0: (codes, scales 2^e)."""
    s = _pow2_scale(_block_max(v, n), qmax)
    return (v / _rows(s, n)[: v.shape[0]]).round().clamp(-qmax, qmax), s


def _per_column(v, bits):
    qmax = 2 ** (bits - 1) - 1
    s = v.abs().amax(0, keepdim=True) / qmax
    return (v / s).round(), s


def _np(t, dtype):
    return t.to(dtype).contiguous().cpu().numpy()


def _e4m3(v):
    return v.to(torch.float8_e4m3fn).view(torch.uint8).contiguous().cpu().numpy()


def _nibbles(codes):
    u = codes.to(torch.int16) & 0xF
    return (u[:, 0::2] | (u[:, 1::2] << 4)).to(torch.uint8).contiguous().cpu().numpy()


def _e2m1_nibbles(v):
    mag = torch.bucketize(v.abs().contiguous(), torch.tensor(_GRID["mxfp4"], device=v.device))
    return _nibbles(mag | (v < 0).to(torch.int64) * 8)


def _layer(g, case, K, N):
    """A layer of N(0, 0.02^2) weights with outlier input channels, split into low-rank factors and quantized residual."""
    main, branch, r = case["main"], case["branch"], case["rank"]
    W = torch.randn(K, N, generator=g, device="cuda") * 0.02
    W[torch.randperm(K, generator=g, device="cuda")[: max(4, K // 100)]] *= 10
    L1q = L2q = s1 = s2 = None
    if r:
        L1 = torch.randn(K, r, generator=g, device="cuda") * 0.05
        L2 = torch.randn(r, N, generator=g, device="cuda") * 0.05
        if branch == "w16a16":
            L1, L2 = L1.half().float(), L2.half().float()
            L1q, L2q = _np(L1, torch.float16), _np(L2, torch.float16)
        elif main in ("mxfp4", "mxint4a8"):
            q = (lambda v: _mxfp(v, branch)) if main == "mxfp4" else (lambda v: _ints(v, 127 if branch == "mxint8" else 7, 32))
            (a, sa), (b, sb) = q(L1), q(L2)
            L1, L2 = a * _rows(sa, 32)[:K], b * _rows(sb, 32)[:r]
            L1q, L2q = (_e4m3(a), _e4m3(b)) if main == "mxfp4" else (_np(a, torch.int8), _np(b, torch.int8))
            s1, s2 = _np(sa, torch.float32), _np(sb, torch.float32)
        else:
            (a, sa), (b, sb) = _per_column(L1, int(branch[1])), _per_column(L2, int(branch[1]))
            L1, L2 = a * sa, b * sb
            L1q, L2q, s1, s2 = _np(a, torch.int8), _np(b, torch.int8), _np(sa[0], torch.float32), _np(sb[0], torch.float32)
        W = W - L1 @ L2
    cfg = B.lq_config_default(K, N, r, branch)
    if main == "sint4":
        s = (_block_max(W, 64) / 7).half().clamp_min(2.0 ** -24)
        packed = _nibbles((W / _rows(s.float(), 64)[:K]).round().clamp(-7, 7))
    else:
        cfg.group = 32
        cfg.main_fmt = {"mxint4": B.MAIN_AUTO, "mxfp4": B.MAIN_MXFP4, "mxint4a8": B.MAIN_MXINT4_A8}[main]
        v, s = _mxfp(W, "mxfp4") if main == "mxfp4" else _ints(W, 7, 32)
        packed = _e2m1_nibbles(v) if main == "mxfp4" else _nibbles(v)
    bias = _np(torch.randn(N, generator=g, device="cuda") * 0.02, torch.float16) if case["bias"] else None
    h = B.lq_layer_import(cfg, packed, _np(s, torch.float16), L1q, s1, L2q, s2, bias)
    B.lq_layer_to_device(h, 0)
    return h


class _Linear:
    """A layer on the GPU with its activation record, an input and the place of its output."""

    def __init__(self, g, case, K, N):
        M, host = case["M"], case["entry"] == "host"
        self.layer = _layer(g, case, K, N)
        self.act = B.lq_act_create(self.layer, M, 0) if case["entry"] != "static" else None
        # unit-variance activations with a few outlier channels; behind an activation function they lean to one side
        x = torch.randn(M, K, generator=g, device="cuda")
        if K > 4000:
            x = torch.nn.functional.gelu(x)
        x[:, torch.randperm(K, generator=g, device="cuda")[: max(8, K // 100)]] *= 20
        dtype = torch.float32 if case["out"] == "f32" else torch.float16
        self.X, self.Y = x.half(), torch.empty(M, N, dtype=dtype, device="cpu" if host else "cuda", pin_memory=host)
        if host:
            self.X = self.X.cpu().pin_memory()

    def __del__(self):
        if getattr(self, "act", None) is not None:
            B.lq_act_free(self.act)
        if getattr(self, "layer", None) is not None:
            B.lq_layer_free(self.layer)


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return {"entry": case["entry"], "M": case["M"], "out": B.OUT_F32 if case["out"] == "f32" else B.OUT_F16,
            "linears": [_Linear(g, case, K, N) for K, N in _shapes(case)]}


def run(state):
    M, out, entry = state["M"], state["out"], state["entry"]
    stream = torch.cuda.current_stream().cuda_stream
    for l in state["linears"]:
        if entry == "device":
            B.lq_quantize_act(l.layer, l.X.data_ptr(), M, l.act, stream)
            B.lq_linear_forward(l.layer, l.act, l.Y.data_ptr(), out, stream)
        elif entry == "static":
            B.lq_linear_forward_static(l.layer, l.X.data_ptr(), M, l.Y.data_ptr(), out, stream)
        else:
            B.lq_linear_forward_host(l.layer, l.act, l.X.data_ptr(), M, l.Y.data_ptr(), out, stream)
    return [l.Y for l in state["linears"]]


def work(case):
    """X in, Y out, the layer once (4-bit codes, block scales, factors at their own width, bias); both products' operations."""
    M, r = case["M"], case["rank"]
    nbytes = flops = 0
    fbits = {"none": 0, "w16a16": 16, "w8a8": 8, "w6a6": 6, "w4a8": 4, "mxfp8": 8, "mxfp6": 6, "mxfp4": 4, "mxint8": 8, "mxint4": 4}[case["branch"]]
    for K, N in _shapes(case):
        scales = -(-K // 64) * N * 2 if case["main"] == "sint4" else -(-K // 32) * N
        nbytes += 2 * M * K + M * N * (4 if case["out"] == "f32" else 2) + K * N // 2 + scales + r * (K + N) * fbits // 8 + 2 * N * case["bias"]
        flops += 2 * M * K * N + 2 * M * r * (K + N)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Codes and scales are exact; only the order of the sums is free.  fp32 output: a few 1e-6 for the integer branches'
    # block sums, 2e-5 where the tensor core sums thousands of products.  fp16 output: one rounding, half an ulp of 2^-10.
    # Where the branch's intermediate is itself a sum in fp32 that is rounded again (to fp16, or to 8-bit blocks whose
    # exponent may move with the block's maximum), two orders of that sum may round apart.
    rel = 1e-5 if case["main"] == "sint4" else 2e-5
    if case["branch"] == "w16a16":
        rel = 3e-4
    elif case["branch"].startswith("mx"):
        rel = 5e-3
    return {"rel": max(rel, 5e-4) if case["out"] == "f16" else rel, "max": 0.05 if rel > 1e-3 else 2e-2 if case["out"] == "f16" or rel > 1e-4 else 1e-3}
