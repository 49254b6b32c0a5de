"""Cases over which the library's speed is followed: the calls a program with LQ-LoRA layers makes.

A layer call is a linear pass over one quantized matrix (forward, input gradient), a training step of one layer (forward,
input gradient, gradients of the two factors from the intermediates the passes leave behind), the forward pass of all
seven matrices of a decoder layer, or the quantization of a matrix.  Shapes, configurations and distributions are those
of ``paper_2311_12023_b200.inputs`` (LLaMA-2-7B / 70B layer shapes, the 8192 x 8192 sweep, the 1024 x 1024 projection).

The calls go through ``paper_2311_12023_b200.binding``.  A program keeps the quantized matrix, the bf16 factors and one
workspace per layer; activations are new in every call and results are returned in fresh tensors.
"""
import math

import torch

from paper_2311_12023_b200 import binding
from paper_2311_12023_b200.inputs import QuantConfig, config_c4_draw


def _case(name, kind, N, K, M, b0, B0, B1, r, weights):
    return {"name": name, "kind": kind, "N": N, "K": K, "M": M, "b0": b0, "B0": B0, "B1": B1, "r": r, "weights": weights}


def listed():
    return [
        # one token through an attention projection of a 7B-sized layer: latency and launches count
        _case("fwd1_4096", "fwd", 4096, 4096, 1, 3, 64, 256, 64, "gaussian"),
        # one token through all seven matrices of a 70B decoder layer with its mixed 2.73-bit configurations
        {"name": "decode1_layer70b", "kind": "layer", "M": 1, "r": 64, "weights": "outliers"},
        # sixteen sequences decoded together, 4-bit codes
        _case("fwd16_8192_nf4", "fwd", 8192, 8192, 16, 4, 64, 256, 64, "gaussian"),
        # input gradient of one position through the 70B down projection (2-bit codes)
        _case("bwd1_8192x28672_nf2", "bwd", 8192, 28672, 1, 2, 128, 256, 64, "outliers"),
        # a short prompt through a small projection (encoder-sized model)
        _case("fwd512_1024", "fwd", 1024, 1024, 512, 3, 64, 256, 64, "gaussian"),
        # a prefill chunk, or a large decode batch
        _case("fwd128_8192", "fwd", 8192, 8192, 128, 3, 64, 256, 64, "gaussian"),
        # fine-tuning on a short sequence of no round length: input gradient of the 7B gate / up projection
        _case("bwd333_11008x4096_nf4", "bwd", 11008, 4096, 333, 4, 64, 256, 64, "student_t"),
        # a training sequence (or prefill) through the 70B gate projection, small blocks: the largest single call
        _case("fwd2048_28672x8192_nf3b16", "fwd", 28672, 8192, 2048, 3, 16, 64, 64, "outliers"),
        # the same length with 8-bit codes
        _case("fwd2048_8192_nf8", "fwd", 8192, 8192, 2048, 8, 64, 256, 64, "gaussian"),
        # fine-tuning step of the 7B down projection: forward, input gradient, factor gradients
        _case("step4096_4096x11008_nf4", "step", 4096, 11008, 4096, 4, 64, 256, 64, "student_t"),
        # quantization of one matrix (run per matrix and configuration by the decomposition and the configuration search)
        _case("encode_8192_nf3", "encode", 8192, 8192, 0, 3, 64, 256, 0, "gaussian"),
        _case("encode_11008x4096_nf4", "encode", 11008, 4096, 0, 4, 64, 256, 0, "student_t"),
    ]


_MAX_FLOPS = 9.0e11       # below the largest listed call
_MAX_WEIGHTS = 28672 * 8192


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "fwd", "bwd", "bwd", "step", "encode"])
    b0 = rng.choice([2, 3, 3, 4, 4, 8])
    B0 = rng.choice([16, 32, 64, 64, 128, 256])
    B1 = rng.choice([64, 256])
    r = rng.choice([0, 16, 64, 64, 64, 128]) if kind in ("fwd", "bwd") else rng.choice([16, 64, 64, 128])
    weights = rng.choice(["gaussian", "student_t", "outliers"])
    step = max(64, B0)
    while True:
        # output columns: any multiple of 8; input columns: whole blocks
        N = 8 * _log_uniform(rng, 128, 28672 // 8)
        K = step * max(1, _log_uniform(rng, 1024, 28672) // step)
        if N * K <= _MAX_WEIGHTS:
            break
    if rng.random() < 0.4:
        N = (N + 127) // 128 * 128 if N <= 28544 else 28672
        if N * K > _MAX_WEIGHTS:
            N = _MAX_WEIGHTS // K // 128 * 128
    if kind == "encode":
        return dict(kind=kind, N=N, K=K, M=0, b0=b0, B0=B0, B1=B1, r=0, weights=weights)
    lo, hi = rng.choice([(1, 16), (17, 512), (512, 4096)]) if kind != "step" else (128, 4096)
    passes = 3 if kind == "step" else 1
    hi = max(lo, min(hi, int(_MAX_FLOPS / (2.0 * passes * N * K))))
    return dict(kind=kind, N=N, K=K, M=_log_uniform(rng, lo, hi), b0=b0, B0=B0, B1=B1, r=r, weights=weights)


# ------------------------------------------------------------------------------------------------ inputs
def _matrices(case):
    """[(N, K, config)] of the case: one matrix, or the seven of the decoder layer."""
    if case["kind"] == "layer":
        return [(m.N, m.K, m.cfg) for m in config_c4_draw()]
    return [(case["N"], case["K"], QuantConfig(case["b0"], case["B0"], 8, case["B1"], 32))]


def _weights(g, N, K, kind):
    """fp32 [N, K] with standard deviation 0.02 (outliers: one entry in a thousand ten times as large)."""
    A = torch.randn(N, K, generator=g, device="cuda")
    if kind == "outliers":
        A *= 0.02
        A[torch.rand(N, K, generator=g, device="cuda") < 0.001] *= 10.0
    elif kind == "student_t":
        chi = torch.zeros_like(A)
        for _ in range(5):
            chi.add_(torch.randn(N, K, generator=g, device="cuda").square_())
        A.div_(chi.div_(5.0).sqrt_()).mul_(0.02 / math.sqrt(5.0 / 3.0))
    else:
        A *= 0.02
    return A


def _bf16(g, rows, cols, std):
    return torch.randn(rows, cols, generator=g, device="cuda").mul_(std).to(torch.bfloat16)


def _inputs(case, seed):
    """Everything the call reads, from the seed alone: per matrix (W, L1, L2, X, dY)."""
    out = []
    for i, (N, K, _) in enumerate(_matrices(case)):
        g = torch.Generator(device="cuda")
        g.manual_seed(1000 * int(seed) + i)
        M, r, kind = case["M"], case["r"], case["kind"]
        W = _weights(g, N, K, case["weights"])
        L1 = _bf16(g, N, r, 0.01) if r else None
        L2 = _bf16(g, r, K, 0.01) if r else None
        X = _bf16(g, M, K, 1.0) if kind in ("fwd", "step", "layer") else None
        dY = _bf16(g, M, N, 1.0) if kind in ("bwd", "step") else None
        out.append((W, L1, L2, X, dY))
        del W
    return out


def prepare(case, seed):
    kind, r, M = case["kind"], case["r"], case["M"]
    mats = _matrices(case)
    if kind == "encode":
        (N, K, cfg), = mats
        W = _inputs(case, seed)[0][0]
        ws = torch.empty(max(16, binding.packed_sizes(N, K, cfg)[3]), dtype=torch.uint8, device="cuda")
        return {"kind": kind, "W": W, "cfg": cfg, "ws": ws}
    layers = []
    for (N, K, cfg), (W, L1, L2, X, dY) in zip(mats, _inputs(case, seed)):
        q = binding.encode(W, cfg)
        del W
        layer = {"q": q, "L1": L1, "L2": L2, "X": X, "dY": dY, "ws": binding.alloc_workspace(q, r, M)}
        if kind == "step":
            layer["ws2"] = binding.alloc_workspace(q, r, M)
            layer["ws3"] = torch.empty(256, dtype=torch.uint8, device="cuda")
        layers.append(layer)
    torch.cuda.empty_cache()
    return {"kind": kind, "r": r, "M": M, "layers": layers}


def run(state):
    kind = state["kind"]
    if kind == "encode":
        q = binding.encode(state["W"], state["cfg"], workspace=state["ws"])
        return [q.codes, q.scale_codes, q.scale2]
    if kind == "layer":
        return [binding.linear_fwd(m["q"], m["L1"], m["L2"], m["X"], workspace=m["ws"]) for m in state["layers"]]
    m, = state["layers"]
    q, L1, L2 = m["q"], m["L1"], m["L2"]
    if kind == "fwd":
        return binding.linear_fwd(q, L1, L2, m["X"], workspace=m["ws"])
    if kind == "bwd":
        return binding.linear_bwd_input(q, L1, L2, m["dY"], workspace=m["ws"])
    r, M = state["r"], state["M"]
    Y = binding.linear_fwd(q, L1, L2, m["X"], workspace=m["ws"])
    dX = binding.linear_bwd_input(q, L1, L2, m["dY"], workspace=m["ws2"])
    T = binding.linear_intermediate(m["ws"], q.N, q.K, q.cfg, r, M, False)
    Tp = binding.linear_intermediate(m["ws2"], q.N, q.K, q.cfg, r, M, True)
    dL1, dL2 = binding.lora_grads_from(T, Tp, q.N, q.K, m["X"], m["dY"], workspace=m["ws3"])
    return [Y, dX, dL1, dL2]


# ------------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    M, r, kind = case["M"], case["r"], case["kind"]
    nbytes = flops = 0
    for N, K, c in _matrices(case):
        packed = N * K * (c.b0 + c.b1 / c.B0 + c.b2 / (c.B0 * c.B1)) / 8
        if kind == "encode":
            # a division, and one comparison per bit of the code; counted as one operation each
            nbytes += 4 * N * K + packed
            flops += N * K * (1 + c.b0)
            continue
        factors = 2 * r * (N + K)
        linear = 2 * M * (N * K + r * K + N * r)
        if kind == "step":
            nbytes += packed + factors + 2 * 2 * M * (N + K) + 2 * factors     # X, dY, Y, dX; fp32 gradients
            flops += 2 * linear + 2 * M * r * (N + K)
        else:
            nbytes += packed + factors + 2 * M * (N + K)
            flops += linear
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    """Codes, scale codes and second-level scales are defined bit for bit.  Linear results: weights and rank-r
    intermediates rounded to bf16, bf16 result: 2.4e-3 from the unrounded layer (measured); a few times that."""
    if case["kind"] == "encode":
        return "exact"
    return {"rel": 1e-2, "max": 5e-2}


# ------------------------------------------------------------------------------------------------ 64-bit values
def _codebook(b0):
    """NormalFloat code book: quantiles of the normal distribution at 2^(b0-1) evenly spaced probabilities below one half
    and 2^(b0-1) + 1 from one half on, divided by the largest, stored in fp32."""
    delta = 0.5 * (1 / 30 + 1 / 32)
    neg = torch.linspace(delta, 0.5, 2 ** (b0 - 1), dtype=torch.float64)
    pos = torch.linspace(0.5, 1 - delta, 2 ** (b0 - 1) + 1, dtype=torch.float64)
    p = torch.cat([neg[:-1], pos])
    z = torch.special.ndtri(p)
    z[2 ** (b0 - 1) - 1] = 0.0
    return (z / z.max()).float().cuda()


def _dequantized(W, cfg):
    """fp64 [N, K]: the quantized matrix, without rounding the products of code-book value and scale."""
    N, K = W.shape
    cb = _codebook(cfg.b0)
    mid = (cb[1:].double() + cb[:-1].double()) / 2
    blocks = W.reshape(-1, cfg.B0)
    s = blocks.abs().amax(dim=1)
    n = s.numel()
    pad = (-n) % cfg.B1
    v = torch.nn.functional.pad(s, (0, pad)).reshape(-1, cfg.B1).amax(dim=1)
    sigma = v / 127.0
    per_block = sigma.repeat_interleave(cfg.B1)[:n]
    sc = torch.where(per_block > 0, (s / per_block).round().clamp(0, 127), torch.zeros_like(s))
    st = sc.double() * per_block.double()
    out = torch.empty(n, cfg.B0, dtype=torch.float64, device=W.device)
    for i in range(0, n, 1 << 20):
        j = min(n, i + (1 << 20))
        sb = s[i:j, None]
        x = torch.where(sb > 0, blocks[i:j] / sb, torch.zeros_like(blocks[i:j]))
        out[i:j] = cb.double()[torch.bucketize(x.double(), mid)] * st[i:j, None]
    return out.reshape(N, K)


def exact(case, seed):
    if case["kind"] == "encode":
        return None
    out = []
    for (N, K, cfg), (W, L1, L2, X, dY) in zip(_matrices(case), _inputs(case, seed)):
        D = _dequantized(W, cfg)
        del W
        if case["r"]:
            l1, l2 = L1.double(), L2.double()
        if X is not None:
            x = X.double()
            t = x @ l2.T if case["r"] else None
            out.append(x @ D.T + (t @ l1.T if case["r"] else 0.0))
        if dY is not None:
            g = dY.double()
            tp = g @ l1 if case["r"] else None
            out.append(g @ D + (tp @ l2 if case["r"] else 0.0))
        if case["kind"] == "step":
            out += [g.T @ t, tp.T @ x]
    return out if case["kind"] in ("layer", "step") else out[0]
