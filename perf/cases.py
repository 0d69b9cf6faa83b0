"""The work a user of this package has it do, as cases that can be timed: the runtime linear layer (activation
quantizer + W4A4 GEMM) from a small layer to the widest one at the largest token count, the same GEMM behind its two
fused producers (norm + reordering, Hadamard + reordering), the offline calibration pass of a layer in NVFP4 and in
integer formats, and the integer fake-quant.  Sizes are those of the package's own layer configurations and token
sweep, plus ragged ones between them.

A case is a dict of plain values; `kind` names the path:
  linear     pipeline.QuantLinear on X [M, K] -> Y [M, N]
  norm       binding.pq_norm_quant_nvfp4 (RMSNorm or adaptive LayerNorm, optional order) + binding.pq_gemm_w4a4
  hadamard   pipeline.QuantLinearH on X [M, K] -> Y [M, N]
  calibrate  pipeline.calibrate over `batches` batches of [M, K] and the weight [N, K]
  fakequant  binding.pq_fakequant_int on [M, K], with or without an order
"""
import math

import torch

from paper_2605_09503_b200 import binding as B
from paper_2605_09503_b200 import pipeline

EPS = 1e-6


def listed():
    return [
        # the small layer of the smoke check: launches and host work are what counts
        dict(name="linear_tiny", kind="linear", M=256, K=512, N=512, gelu=False),
        # text stream of a DiT block (512 tokens): a fraction of the chip's tiles
        dict(name="linear_text_out", kind="linear", M=512, K=3072, N=3072, gelu=False),
        # an image of an odd number of tokens through a layer whose width is no multiple of a tile
        dict(name="linear_ragged", kind="linear", M=1357, K=1088, N=4312, gelu=False),
        # attention QKV projection, 4096 image + 512 text tokens: the ordinary call of the runtime path
        dict(name="linear_qkv", kind="linear", M=4608, K=3072, N=9216, gelu=False),
        # MLP down-projection: long K, GELU activations
        dict(name="linear_mlp_down", kind="linear", M=4608, K=12288, N=3072, gelu=True),
        # MLP up-projection at the largest token count of the sweep
        dict(name="linear_mlp_up_18432", kind="linear", M=18432, K=3072, N=12288, gelu=False),
        # adaptive LayerNorm with the channel order absorbed into it, in front of the QKV projection
        dict(name="norm_adaln_qkv", kind="norm", M=4608, K=3072, N=9216, rms=False, order=True),
        # Hadamard variant of the attention output projection
        dict(name="hadamard_out", kind="hadamard", M=4608, K=3072, N=3072),
        # offline pass of the small layer, integer format: many small launches
        dict(name="calibrate_tiny", kind="calibrate", M=256, K=512, N=512, batches=4, bits=4, group=32),
        # offline pass of the QKV projection, NVFP4 errors (bits 0), eight calibration batches
        dict(name="calibrate_qkv", kind="calibrate", M=4608, K=3072, N=9216, batches=8, bits=0, group=16),
        # one layer of the integer acceptance sweep
        dict(name="calibrate_int4_g64", kind="calibrate", M=4608, K=3072, N=3072, batches=1, bits=4, group=64),
        # integer quantize-dequantize of reordered activations (simulated W4A4)
        dict(name="fakequant_int4_g64", kind="fakequant", M=4608, K=3072, bits=4, group=64, order=True),
    ]


_MAX_GEMM = 18432 * 3072 * 12288            # the largest listed linear layer
_MAX_CALIB = (8 * 4608 + 9216) * 3072       # the largest listed calibration


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, step):
    return max(lo, min(hi, step * int(round(_log(rng, lo, hi) / step))))


def draw(rng):
    """One more case of the same ranges: odd token counts, widths at the granularity the entry points take."""
    kind = rng.choice(["linear"] * 8 + ["norm"] * 3 + ["hadamard"] * 2 + ["calibrate"] * 3 + ["fakequant"] * 2)
    if kind == "fakequant":
        group = rng.choice([32, 64, 128])
        K = _width(rng, 512, 12288, group)
        return dict(kind=kind, M=_log(rng, 256, min(18432, 18432 * 3072 // K)), K=K, bits=rng.choice([3, 4]), group=group,
                    order=rng.random() < 0.5)
    if kind == "calibrate":
        bits = rng.choice([0, 0, 3, 4])
        group = 16 if bits == 0 else rng.choice([32, 64, 128])
        K = _width(rng, 512, 12288, max(group, 64))
        N = _width(rng, 512, min(9216, _MAX_CALIB // (2 * K)), 8)
        batches = rng.randint(1, 8)
        M = _log(rng, 128, max(129, min(4608, (_MAX_CALIB // K - N) // batches)))
        return dict(kind=kind, M=M, K=K, N=N, batches=batches, bits=bits, group=group)
    if kind == "hadamard":
        K = rng.choice([768, 1024, 1536, 2048, 3072, 3072, 4096, 6144, 12288])
    elif kind == "norm":
        K = _width(rng, 512, 6144, 64)
    else:
        K = _width(rng, 512, 12288, 64)
    N = _width(rng, 512, 12288, 8)
    M = _log(rng, 128, min(18432 if kind == "linear" else 9216, _MAX_GEMM // (K * N)))
    case = dict(kind=kind, M=M, K=K, N=N)
    if kind == "linear":
        case["gelu"] = rng.random() < 0.25
    if kind == "norm":
        case["rms"], case["order"] = rng.random() < 0.5, rng.random() < 0.75
    return case


# ------------------------------------------------------------------------------------------------- inputs
def _activations(g, rows, K, scale, gelu=False):
    x = torch.randn(rows, K, device="cuda", generator=g)
    if gelu:
        x = torch.nn.functional.gelu(x)
    return (x * scale).to(torch.bfloat16)


def _channel_scale(g, K, sigma=1.5, outliers=True):
    """Log-normal channel scales, one channel in a hundred fifty times larger."""
    scale = torch.exp(sigma * torch.randn(K, device="cuda", generator=g))
    if outliers:
        scale[torch.randperm(K, device="cuda", generator=g)[:max(1, K // 100)]] *= 50.0
    return scale


def _weight(g, N, K, std=0.02):
    return (std * torch.randn(N, K, device="cuda", generator=g)).to(torch.bfloat16)


def _hadamard(x, dtype):
    """x (H_m (x) H_{2^n}) / sqrt(K) of every row, K = m 2^n with m = 1 or 12 (Paley's matrix of order 12)."""
    M, K = x.shape
    m = 12 if K % 3 == 0 else 1
    y = x.to(dtype).view(M, m, K // m)
    if m == 12:
        squares = {i * i % 11 for i in range(1, 11)}
        H = torch.eye(12, dtype=dtype)
        for i in range(12):
            for j in range(12):
                if i != j:
                    H[i, j] = 1.0 if i == 0 else -1.0 if j == 0 else (1.0 if (i - j) % 11 in squares else -1.0)
        y = torch.einsum("rab,ac->rcb", y, H.to(x.device))
    stride = 1
    while stride < K // m:
        y = y.reshape(M, -1, 2, stride)
        y = torch.stack((y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]), 2)
        stride *= 2
    return y.reshape(M, K) / math.sqrt(K)


def _tensor_scale(t):
    return (t.abs().amax().float() / 2688.0).reshape(1)


def _order(g, K):
    return torch.randperm(K, device="cuda", generator=g).to(torch.int32)


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind, M, K = case["kind"], case["M"], case["K"]
    scale = _channel_scale(g, K, 2.0 if case.get("gelu") else 1.5, not case.get("gelu"))
    t = dict(order=None)
    if kind == "calibrate":
        t["batches"] = [_activations(g, M, K, scale) for _ in range(case["batches"])]
    else:
        t["X"] = _activations(g, M, K, scale, case.get("gelu", False))
    if kind == "fakequant":
        t["order"] = _order(g, K) if case["order"] else None
        return t
    t["W"] = _weight(g, case["N"], K)
    if kind == "linear":
        t["ts_x"] = _tensor_scale(t["X"])
    elif kind == "hadamard":
        t["ts_x"] = _tensor_scale(_hadamard(t["X"], torch.float32))
        t["order"] = _order(g, K)
    elif kind == "norm":
        rms = case["rms"]
        t["a"] = 1.0 + 0.2 * torch.randn(K, device="cuda", generator=g) if rms else 0.2 * torch.randn(K, device="cuda", generator=g)
        t["b"] = None if rms else 0.2 * torch.randn(K, device="cuda", generator=g)
        t["order"] = _order(g, K) if case["order"] else None
        x = t["X"].float()
        t["ts_x"] = _tensor_scale(x / (x.square().mean(1, keepdim=True) + EPS).sqrt())  # stands in for the calibrated scale
    return t


def _format(case):
    return pipeline.NVFP4 if case["bits"] == 0 else (B.KIND_INT, case["bits"], case["group"])


def prepare(case, seed):
    """Inputs, quantized weight and layer object a program holds before the call."""
    kind, M, K = case["kind"], case["M"], case["K"]
    t = _inputs(case, seed)
    if kind == "fakequant":
        return dict(kind=kind, X=t["X"], fmt=_format(case), order=t["order"], out=torch.empty_like(t["X"]))
    if kind == "calibrate":
        return dict(kind=kind, batches=t["batches"], W=t["W"], fmt=_format(case))
    N = case["N"]
    wq = torch.empty(N, K // 2, dtype=torch.uint8, device="cuda")
    sfw = torch.empty(B.sf_bytes(N, K, B.PQ_SF_TCGEN05), dtype=torch.uint8, device="cuda")
    ts_w = torch.empty(1, dtype=torch.float32, device="cuda")
    B.pq_quant_weight(t["W"], None, None, wq, sfw, B.PQ_SF_TCGEN05, ts_w, B.workspace(B.OP_QUANT_WEIGHT, N, K))
    if kind == "linear":
        return dict(kind=kind, X=t["X"], layer=pipeline.QuantLinear(wq, sfw, ts_w, t["ts_x"], M))
    if kind == "hadamard":
        return dict(kind=kind, X=t["X"], layer=pipeline.QuantLinearH(wq, sfw, ts_w, t["ts_x"], M, t["order"]))
    return dict(kind=kind, H=t["X"], norm=B.NORM_RMS if case["rms"] else B.NORM_ADALN, a=t["a"], b=t["b"], order=t["order"],
                ts_x=t["ts_x"], codes=torch.empty(M, K // 2, dtype=torch.uint8, device="cuda"),
                sf=torch.empty(B.sf_bytes(M, K, B.PQ_SF_TCGEN05), dtype=torch.uint8, device="cuda"),
                wq=wq, sfw=sfw, ts_w=ts_w, Y=torch.empty(M, N, dtype=torch.bfloat16, device="cuda"),
                ws=B.workspace(B.OP_GEMM, M, K, N))


def run(state):
    kind = state["kind"]
    if kind in ("linear", "hadamard"):
        return state["layer"](state["X"])
    if kind == "norm":
        B.pq_norm_quant_nvfp4(state["H"], state["norm"], state["a"], state["b"], EPS, state["order"], state["ts_x"],
                              state["codes"], state["sf"], B.PQ_SF_TCGEN05)
        B.pq_gemm_w4a4(state["codes"], state["sf"], state["ts_x"], state["wq"], state["sfw"], state["ts_w"], state["Y"], state["ws"])
        return state["Y"], state["codes"], state["sf"]
    if kind == "fakequant":
        B.pq_fakequant_int(state["X"], state["fmt"], state["order"], state["out"])
        return state["out"]
    c = pipeline.calibrate(state["batches"], state["W"], fmt=state["fmt"])
    return dict(sumsq_a=c.sumsq_a, sumsq_w=c.sumsq_w, amax_a=c.amax_a, ts_x=c.ts_x, ts_w=c.ts_w, perms=c.perms, err_x=c.err_x,
                err_w=c.err_w, lam=c.lam, E=c.E, select=c.select, wq=c.wq, sfw=c.sfw)


# ------------------------------------------------------------------------------------------------- the same in 64 bits
# The quantizers are defined in fp32 (scale = E4M3 or fp32 quotient, one reciprocal, one product per element), so a code
# is taken from these operations; everything that is a sum, a product of decoded values or a transform is float64.
_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _decoded(x, ts, fmt):
    """Quantized-dequantized values of fp32 rows x: (levels, decode scales), both float64, groups along the last dim."""
    _, bits, group = fmt
    xg = x.view(x.shape[0], -1, group)
    amax = xg.abs().amax(-1, keepdim=True)
    if fmt[0] == B.KIND_INT:
        Q = float((1 << (bits - 1)) - 1)
        d = amax / Q
        z = torch.round(xg * torch.where(d > 0, 1.0 / d, 0.0)).clamp(-Q, Q)
    else:
        sf = (amax / (6.0 * ts)).clamp(max=448.0).to(torch.float8_e4m3fn).float()
        d = sf * ts
        y = xg * torch.where(d > 0, 1.0 / d, 0.0)
        grid = torch.tensor(_E2M1, device=x.device)
        mid = (grid[1:] + grid[:-1]) / 2
        mag = y.abs().contiguous()
        # nearest level; a midpoint goes to the code with the even number
        lower, upper = torch.bucketize(mag, mid), torch.bucketize(mag, mid, right=True)
        z = torch.where(y < 0, -1.0, 1.0) * grid[torch.where(upper % 2 == 0, upper, lower)]
    return z.double(), d.double()


def _decode(x, ts, fmt):
    z, d = _decoded(x, ts, fmt)
    return (z * d).view(x.shape)


def _weight_ts(W):
    return (W.abs().amax().float() / 2688.0).reshape(1)


def _tensor_errors(x, ts, fmt, perms):
    """Sum over the rows of the squared group errors, original order first, then every candidate: float64 [P + 1, K / g]."""
    err = []
    for perm in [None] + list(perms):
        total = 0
        for rows in x.split(4608):
            v = (rows if perm is None else rows[:, perm.long()]).float()
            z, d = _decoded(v, ts, fmt)
            total = total + (v.double().view(z.shape) - z * d).square().sum((0, 2))
        err.append(total)
    return torch.stack(err)


def exact(case, seed):
    """What run returns for these inputs in float64; whole values (codes, scale bytes, orders, decisions) have no such value."""
    t = _inputs(case, seed)
    kind, K = case["kind"], case["K"]
    if kind == "fakequant":
        x = t["X"] if t["order"] is None else t["X"][:, t["order"].long()]
        return _decode(x.float(), None, _format(case))
    W = t["W"]
    if kind == "calibrate":
        fmt, J = _format(case), 5
        x = torch.cat(t["batches"])
        sa = sum(b.double().square().sum(0) for b in t["batches"])
        sw = W.double().square().sum(0)
        amax = x.abs().amax(0).float()
        ts_x, ts_w = (amax.amax() / 2688.0).reshape(1), _weight_ts(W)
        a, w = sa / x.shape[0], sw / W.shape[0]
        perms = torch.stack([torch.argsort(a ** j * w ** (J - j), descending=True, stable=True) for j in range(J + 1)])
        err_x, err_w = _tensor_errors(x, ts_x, fmt, perms), _tensor_errors(W, ts_w, fmt, perms)
        lam = torch.stack((1.0 / sa.sum(), 1.0 / sw.sum()))
        return dict(sumsq_a=sa, sumsq_w=sw, amax_a=amax.double(), ts_x=ts_x.double(), ts_w=ts_w.double(), perms=None, err_x=err_x,
                    err_w=err_w, lam=lam, E=lam[0] * err_x.sum(1) + lam[1] * err_w.sum(1), select=None, wq=None, sfw=None)
    x = t["X"]
    if kind == "hadamard":
        x = _hadamard(x, torch.float64)
    elif kind == "norm":
        x = x.double()
        if case["rms"]:
            x = x / (x.square().mean(1, keepdim=True) + EPS).sqrt()
        else:
            x = (x - x.mean(1, keepdim=True)) / (x.var(1, unbiased=False, keepdim=True) + EPS).sqrt()
    if t["order"] is not None:
        x = x[:, t["order"].long()]
    if kind == "norm":
        x = x * t["a"].double() if case["rms"] else x * (1.0 + t["a"].double()) + t["b"].double()
    wd = _decode(W.float(), _weight_ts(W), pipeline.NVFP4).T
    y = torch.cat([_decode(rows.float().contiguous(), t["ts_x"], pipeline.NVFP4) @ wd for rows in x.split(4608)])
    return (y, None, None) if kind == "norm" else y


# ------------------------------------------------------------------------------------------------- what a pass cannot do without
def _codes_bytes(rows, K):
    return rows * K // 2 + rows * K // 16


def work(case):
    kind, M, K = case["kind"], case["M"], case["K"]
    if kind == "fakequant":
        return {"bytes": 4 * M * K + (4 * K if case["order"] else 0), "flops": 4 * M * K}
    N = case["N"]
    if kind == "calibrate":
        rows = M * case["batches"] + N
        groups = K // case["group"]
        # every tensor once; the sums of squares, and of seven orders scaling, residual and square per element
        return {"bytes": 2 * rows * K + _codes_bytes(N, K) + 6 * 4 * K + 2 * 7 * 8 * groups + 20 * K,
                "flops": (2 + 7 * 5) * rows * K}
    flops = 2 * M * N * K
    extra = {"linear": 0, "norm": 6 * M * K, "hadamard": M * K * int(math.log2(K))}[kind]
    out_codes = _codes_bytes(M, K) if kind == "norm" else 0
    return {"bytes": 2 * M * K + out_codes + _codes_bytes(N, K) + 2 * M * N, "flops": flops + extra}


def tolerance(case):
    """Codes, scale bytes, orders, decisions and the offline sums have one right answer (the order of their additions is part
    of the interface).  A product is the bf16 rounding of an fp32 sum whose order is free: against a float64 product rounded
    to bf16, and against fp32 sums taken in eight slices of K, the listed layers differ by 1e-6 to 3.3e-5 (2-norm) and by one
    bf16 step (0.0078) where a sum lies at a rounding boundary; about four times that is allowed."""
    if case["kind"] in ("calibrate", "fakequant"):
        return "exact"
    return {"rel": 1.5e-4, "max": 0.03, "differ": 0.0}
