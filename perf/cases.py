"""The work that a user of this library has it do, as measurable cases.

Four kinds of call, each through the public binding:

  compress  a weight matrix in host memory -> codebook, codes (and the decoded matrix): cc_compress_host
  fit       sub-vectors already on the device -> Lloyd iterations, then the FP16 codebook and its codes:
            cc_set_codebook, cc_fit, cc_finalize
  decode    codes -> weight matrix: cc_decode
  grad      gradient of the loss with respect to the weight -> gradient with respect to the codebook
            (training with the codes fixed): cc_reshape_subvectors, cc_codebook_grad
  linear    forward of the compressed layer, FP16 codebook or the 4-bit one: cc_linear_forward(_q4)

Weights are heavy-tailed (Student t with three degrees of freedom, a few large outliers), as the
repository's workloads draw them; activations are normal.
"""
from __future__ import annotations

import math

import torch

from paper_2503_13089_b200 import binding as cc

SCALE = 0.02
MOST_SCORES = 8192 * 28672 // 4 * 65536 * 5          # point-centroid pairs of the largest fit
MOST_LINEAR = 4096 * 4096 * 4096                     # multiply-adds of the largest layer forward


def listed():
    return [
        # a small matrix end to end from host memory: bound by latency and the number of launches
        {"name": "compress_256x512_g4", "op": "compress", "d_out": 256, "d_in": 512, "g": 4, "K": 256, "iters": 10, "decode": True},
        # an attention projection with 12-bit codes, decoded copy wanted back
        {"name": "compress_4096_g4_k4096", "op": "compress", "d_out": 4096, "d_in": 4096, "g": 4, "K": 4096, "iters": 20, "decode": True},
        # the same matrix in the 3-bit setting of the paper: padded out_features, odd codebook size
        {"name": "compress_4096_g6_k65500", "op": "compress", "d_out": 4096, "d_in": 4096, "g": 6, "K": 65500, "iters": 20, "decode": False},
        # an MLP matrix at 2 bits a weight
        {"name": "fit_11008_g8_k65536", "op": "fit", "d_out": 11008, "d_in": 4096, "g": 8, "K": 65536, "iters": 20},
        # an MLP matrix of a large model at 4 bits a weight (a few of its iterations)
        {"name": "fit_28672_g4_k65536", "op": "fit", "d_out": 8192, "d_in": 28672, "g": 4, "K": 65536, "iters": 5},
        # one bit a weight: few points for each centroid
        {"name": "fit_4096_g16_k65536", "op": "fit", "d_out": 4096, "d_in": 4096, "g": 16, "K": 65536, "iters": 15},
        # weights rebuilt from their codes
        {"name": "decode_28672_g4_k65536", "op": "decode", "d_out": 8192, "d_in": 28672, "g": 4, "K": 65536},
        # backward: a training step's gradient with respect to the codebook
        {"name": "grad_4096_g4_k65536", "op": "grad", "d_out": 4096, "d_in": 4096, "g": 4, "K": 65536},
        # generation, one token, on the codebook as stored and on the 4-bit one
        {"name": "linear_1_g4_k65536", "op": "linear", "M": 1, "d_out": 4096, "d_in": 4096, "g": 4, "K": 65536, "q4": False, "bias": False},
        {"name": "linear_q4_1_g4_k65536", "op": "linear", "M": 1, "d_out": 4096, "d_in": 4096, "g": 4, "K": 65536, "q4": True, "bias": False},
        # generation for a batch, padded out_features, with a bias
        {"name": "linear_33_g6_k65500", "op": "linear", "M": 33, "d_out": 11008, "d_in": 4096, "g": 6, "K": 65500, "q4": False, "bias": True},
        # a prompt
        {"name": "linear_4096_g4_k65536", "op": "linear", "M": 4096, "d_out": 4096, "d_in": 4096, "g": 4, "K": 65536, "q4": False, "bias": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A matrix edge: mostly a multiple of 64 as layers have, sometimes any number."""
    v = _log(rng, lo, hi)
    return v if rng.random() < 0.25 else max(64, v // 64 * 64)


def _subvectors(d_out, d_in, g):
    return d_in * ((d_out + g - 1) // g)


def draw(rng):
    op = rng.choice(["compress", "fit", "fit", "decode", "grad", "linear", "linear", "linear"])
    g = rng.choice([4, 4, 5, 6, 7, 8, 9, 16])
    if op in ("compress", "fit"):
        while True:
            hi = 8192 if op == "compress" else 28672
            c = {"op": op, "d_out": _size(rng, 256, hi), "d_in": _size(rng, 256, hi), "g": g,
                 "K": min(65536, _log(rng, 256, 80000)), "iters": rng.randint(5, 20)}
            N = _subvectors(c["d_out"], c["d_in"], g)
            dear = 1.0 if g <= 7 else 1.7                # a longer contraction
            if 4 * c["K"] <= N <= 60000000 and N * c["K"] * c["iters"] * dear <= MOST_SCORES:
                break
        if op == "compress":
            c["decode"] = rng.random() < 0.5
        return c
    if op in ("decode", "grad"):
        while True:
            c = {"op": op, "d_out": _size(rng, 256, 28672), "d_in": _size(rng, 256, 28672), "g": g,
                 "K": min(65536, _log(rng, 256, 80000))}
            if c["K"] <= _subvectors(c["d_out"], c["d_in"], g) <= 60000000 and c["d_out"] * c["d_in"] <= 8192 * 28672:
                return c
    while True:
        M = _log(rng, 1, 4096)
        q4 = rng.random() < 0.4
        if q4:
            g = rng.choice([4, 4, 6, 8, 16])
        K = min(65536, _log(rng, 1024, 80000))
        c = {"op": "linear", "M": M, "d_out": _size(rng, 512, 11008), "d_in": _size(rng, 512, 11008), "g": g,
             "K": min(K, 262144 // g) if q4 else K, "q4": q4, "bias": rng.random() < 0.5}
        if M * c["d_out"] * c["d_in"] <= MOST_LINEAR:
            return c


# ------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _heavy(n, gen, scale=SCALE, outliers=5e-4):
    """n FP16 values: scale * t(3), a share of them replaced by +-U(0.2, 1)."""
    out = torch.empty(n, dtype=torch.float16, device="cuda")
    step = 1 << 25
    for lo in range(0, n, step):
        m = min(step, n - lo)
        z = torch.randn(m, device="cuda", generator=gen)
        chi = torch.randn(m, device="cuda", generator=gen).square_()
        chi += torch.randn(m, device="cuda", generator=gen).square_()
        chi += torch.randn(m, device="cuda", generator=gen).square_()
        z *= torch.rsqrt(chi.mul_(1.0 / 3.0).clamp_(min=1e-12)).mul_(scale)
        if outliers:
            u = torch.rand(m, device="cuda", generator=gen)          # below `outliers`: replaced, magnitude and sign from u
            v = torch.rand(m, device="cuda", generator=gen).mul_(1.6).sub_(0.8)
            z = torch.where(u < outliers, v + v.sign() * 0.2, z)
        out[lo:lo + m] = z.clamp_(-65504, 65504).to(torch.float16)
    return out


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


_context = None


def _ctx():
    """One context for the process, as a program that compresses or serves a whole model keeps one."""
    global _context
    if _context is None:
        _context = cc.Context(torch.cuda.current_device())
    return _context


def prepare(case, seed):
    gen = _gen(seed)
    op, g, K = case["op"], case["g"], case["K"]
    d_out, d_in = case["d_out"], case["d_in"]
    N = _subvectors(d_out, d_in, g)
    s = dict(case, ctx=_ctx(), N=N)
    dev = "cuda"
    if op == "compress":
        s["W"] = _pinned(_heavy(d_out * d_in, gen).view(d_out, d_in))
        s["C16"] = torch.empty((K, g), dtype=torch.float16, pin_memory=True)
        s["idx"] = torch.empty(N, dtype=torch.uint16, pin_memory=True)
        s["trace"] = torch.empty(case["iters"] + 1, dtype=torch.float64, pin_memory=True)
        s["W_hat"] = torch.empty((d_out, d_in), dtype=torch.float16, pin_memory=True) if case["decode"] else None
        s["seed"] = seed
        return s
    if op == "fit":
        s["ctx"].ensure_workspace(N, g, K)
        W = _heavy(d_out * d_in, gen).view(d_out, d_in)
        s["X"] = torch.empty((N, g), dtype=torch.float16, device=dev)
        cc.cc_reshape_subvectors(s["ctx"], W, d_out, d_in, g, cc.LAYOUT_PAPER_T, s["X"])
        del W
        s["C0"] = torch.empty((K, g), dtype=torch.float32, device=dev)
        cc.cc_init_codebook(s["ctx"], s["X"], N, g, K, seed, s["C0"])
        s["C"] = torch.empty_like(s["C0"])
        s["C16"] = torch.empty((K, g), dtype=torch.float16, device=dev)
        s["idx"] = torch.empty(N, dtype=torch.uint16, device=dev)
        s["dist"] = torch.empty(N, dtype=torch.float32, device=dev)
        s["counts"] = torch.empty(K, dtype=torch.int32, device=dev)
        s["trace"] = torch.empty(case["iters"] + 1, dtype=torch.float64, device=dev)
        return s
    # codes as a clustering of such weights leaves them: all of them in use, the popular ones more often
    s["idx"] = (torch.rand(N, device=dev, generator=gen).square_() * K).clamp_(max=K - 1).to(torch.int32).to(torch.uint16)
    s["C16"] = _heavy(K * g, gen).view(K, g)
    if op == "decode":
        s["W_hat"] = torch.empty((d_out, d_in), dtype=torch.float16, device=dev)
    elif op == "grad":
        s["ctx"].ensure_workspace(N, g, K)
        s["dW"] = _heavy(d_out * d_in, gen, 1e-3, 0.0).view(d_out, d_in)
        s["dX"] = torch.empty((N, g), dtype=torch.float16, device=dev)
        s["dC"] = torch.empty((K, g), dtype=torch.float32, device=dev)
    else:
        M = case["M"]
        s["ctx"].ensure_workspace(1, g, K, at_least=cc.cc_linear_workspace_bytes(s["ctx"], M, d_out, d_in))
        s["x"] = (torch.randn((M, d_in), device=dev, generator=gen) * 0.5).to(torch.float16)
        s["b"] = torch.randn(d_out, device=dev, generator=gen) if case["bias"] else None
        s["y"] = torch.empty((M, d_out), dtype=torch.float32, device=dev)
        if case["q4"]:
            s["q"] = torch.empty((K * g + 1) // 2, dtype=torch.uint8, device=dev)
            s["scale"] = torch.empty(1, dtype=torch.float32, device=dev)
            cc.cc_quantize_codebook(s["ctx"], s["C16"], K, g, 4, s["q"], s["scale"])
    return s


def run(s):
    op, ctx, N, g, K, d_out, d_in = s["op"], s["ctx"], s["N"], s["g"], s["K"], s["d_out"], s["d_in"]
    if op == "compress":
        cc.cc_compress_host(ctx, s["W"], d_out, d_in, g, K, s["iters"], s["seed"], cc.LAYOUT_PAPER_T, s["C16"], s["idx"],
                            s["trace"], s["W_hat"])
        return [s["C16"], s["idx"].view(torch.int16), s["trace"], s["W_hat"]]
    if op == "fit":
        cc.cc_set_codebook(ctx, s["C0"], K, g, s["C"])
        cc.cc_fit(ctx, s["X"], N, g, K, s["iters"], s["C"], s["idx"], s["dist"], s["counts"], s["trace"])
        cc.cc_finalize(ctx, s["X"], N, g, s["C"], K, s["C16"], s["idx"], s["dist"], s["trace"][s["iters"]:])
        return [s["C"], s["C16"], s["idx"].view(torch.int16), s["dist"], s["counts"], s["trace"]]
    if op == "decode":
        cc.cc_decode(ctx, s["C16"], K, g, s["idx"], d_out, d_in, cc.LAYOUT_PAPER_T, s["W_hat"])
        return s["W_hat"]
    if op == "grad":
        cc.cc_reshape_subvectors(ctx, s["dW"], d_out, d_in, g, cc.LAYOUT_PAPER_T, s["dX"])
        cc.cc_codebook_grad(ctx, s["dX"], N, g, s["idx"], K, s["dC"])
        return [s["dX"], s["dC"]]
    if s["q4"]:
        cc.cc_linear_forward_q4(ctx, s["x"], s["M"], s["q"], s["scale"], K, g, s["idx"], d_out, d_in, s["b"], s["y"])
    else:
        cc.cc_linear_forward(ctx, s["x"], s["M"], s["C16"], K, g, s["idx"], d_out, d_in, s["b"], s["y"])
    return s["y"]


def work(case):
    """Each input read once, each output written once.  Operations of the clustering: the distance of every
    point to the centroid it ends up with and its share of that centroid's mean, in every iteration.  How many
    OTHER centroids a method has to look at is the method's affair (a search over all of them: 2 g N K)."""
    op, g, K, d_out, d_in = case["op"], case["g"], case["K"], case["d_out"], case["d_in"]
    N = _subvectors(d_out, d_in, g)
    if op == "compress":
        it = case["iters"] + 1
        by = 2.0 * d_out * d_in + 2.0 * K * g + 2.0 * N + 8.0 * it + (2.0 * d_out * d_in if case["decode"] else 0.0)
        return {"bytes": by, "flops": 4.0 * g * N * it}
    if op == "fit":
        it = case["iters"] + 1
        return {"bytes": 2.0 * N * g + 4.0 * K * g + (4.0 + 2.0) * K * g + 4.0 * K + (2.0 + 4.0) * N + 8.0 * it,
                "flops": 4.0 * g * N * it}
    if op == "decode":
        return {"bytes": 2.0 * N + 2.0 * K * g + 2.0 * d_out * d_in, "flops": 0.0}
    if op == "grad":
        return {"bytes": 2.0 * d_out * d_in + 2.0 * N * g + 2.0 * N + 4.0 * K * g, "flops": 1.0 * N * g}
    M = case["M"]
    book = 0.5 * K * g if case["q4"] else 2.0 * K * g
    return {"bytes": 2.0 * N + book + 2.0 * M * d_in + 4.0 * M * d_out + (4.0 * d_out if case["bias"] else 0.0),
            "flops": 2.0 * M * d_out * d_in}


def tolerance(case):
    """Clustering, decode and codebook gradient: codes, counts, centroids and distances have one right answer in
    the arithmetic that the interface states (exact integer sums, float64 decisions, one rounding), so nothing
    but the order of the objective's float64 sum is free (2e-13 seen).  Layer forward: products are exact, the
    FP32 accumulation is not; the present kernels are LINEAR_SEEN from a float64 product on the same inputs."""
    if case["op"] in ("decode", "grad"):
        return "exact"
    if case["op"] in ("compress", "fit"):
        return {"rel": 1e-12, "max": 1e-12, "differ": 0.0}
    return {"rel": 1e-5, "max": 1e-4}
