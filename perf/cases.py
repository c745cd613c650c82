"""Timed cases of Nystrom Laplacian attention: the calls a training or inference program makes, over the sizes it makes
them at.

Five kinds of call, all through the public entry points:
  train   forward + backward of the attention path (laplace_nystrom_fwd, laplace_nystrom_bwd)
  infer   forward only, no saved context
  block   forward + backward of the attention block (rotary embedding, the path, depth-wise convolution branch)
  solver  ns_pinv + ns_pinv_bwd on a batch of landmark kernel matrices
  kernel  l1_kernel + l1_kernel_bwd on plain token matrices
Inputs are synthetic, with the distributions of paper_2604_20368_b200/synth.py: Q, K, V, dO ~ N(0, sigma^2) in the
storage type, V ~ U(-1, 1) and a tenth of the landmark regions copies of others where `dup` is set, and a constant
whitening scale.  The decay is lambda = d, the ridge 1e-6.
"""
from __future__ import annotations

import math

import torch

import paper_2604_20368_b200 as ln
from paper_2604_20368_b200 import binding

RIDGE = 1e-6


def _path(name, kind, B, H, gh, gw, d, mh, mw, T, prefix=0, dtype="bf16", sigma=1.0, dup=False):
    c = dict(kind=kind, B=B, H=H, gh=gh, gw=gw, d=d, mh=mh, mw=mw, T=T, prefix=prefix, dtype=dtype, sigma=sigma, dup=dup)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # smallest call: one image, three heads, fp32 storage, forward only; a handful of CTAs, so launches and latency
        _path("tiny_infer_f32", "infer", 1, 3, 14, 14, 64, 4, 8, 6, dtype="f32"),
        # DeiT-Small-shaped training step: class token + 14 x 14 patches, many small heads
        _path("deit_train", "train", 64, 6, 14, 14, 64, 7, 7, 6, prefix=1),
        # first stage of a pyramid backbone (PVT): 56 x 56 tokens, one head per image
        _path("pvt1_train", "train", 32, 1, 56, 56, 64, 8, 8, 8),
        # high-resolution training step, 112 x 112 tokens
        _path("hires112_train", "train", 8, 2, 112, 112, 64, 8, 16, 8, sigma=0.5),
        # high-resolution inference, 224 x 224 tokens per head: the longest sequences
        _path("hires224_infer", "infer", 8, 2, 224, 224, 64, 8, 16, 8, sigma=0.5),
        # wide heads, duplicated keys (near-singular landmark matrix), 128 landmarks
        _path("stress_m128_train", "train", 16, 8, 64, 64, 128, 8, 16, 8, dup=True),
        # the largest training step: 256 landmarks and the longest iteration
        _path("stress_m256_train", "train", 16, 8, 64, 64, 128, 16, 16, 12, dup=True),
        # sizes that divide nothing: class token, a 37 x 29 grid pooled to 5 x 7 overlapping regions, three images of five heads
        _path("ragged_train", "train", 3, 5, 37, 29, 128, 5, 7, 5, prefix=1),
        # fp32 storage, the precision a user checks gradients or trains small models in
        _path("f32_train", "train", 8, 4, 28, 28, 64, 7, 7, 6, dtype="f32"),
        # the whole attention block on the pyramid stage's shape: rotary embedding and the 3 x 3 convolution branch
        _path("block_train", "block", 16, 2, 56, 56, 64, 7, 7, 6),
        # the solver on its own, forward and backward: the landmark matrices of a layer's sixteen heads
        dict(name="solver_m128", kind="solver", batch=16, m=128, T=8, d=64),
        # the kernel block on its own, forward and backward: two heads, 32 channels, 1024 x 1024 pairs
        dict(name="kernel_1024", kind="kernel", batch=2, na=1024, nb=1024, d=32, dtype="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train", "infer", "infer", "block", "solver", "kernel"])
    if kind == "solver":
        m = rng.randint(16, 256)
        return dict(kind=kind, batch=_log_int(rng, 1, max(2, 64 * 128 // m)), m=m, T=rng.randint(4, 12), d=rng.choice([32, 64, 128]))
    if kind == "kernel":
        return dict(kind=kind, batch=rng.randint(1, 4), na=_log_int(rng, 64, 3000), nb=_log_int(rng, 64, 3000),
                    d=rng.choice([32, 64, 128]), dtype=rng.choice(["f32", "bf16"]))
    d = rng.choice([32, 64, 64, 64, 128, 128])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    gh = _log_int(rng, 8, 224 if dtype == "bf16" else 64)
    gw = min(224, max(8, int(round(gh * rng.uniform(0.7, 1.4)))))
    mh, mw = _log_int(rng, 2, min(16, gh)), _log_int(rng, 2, min(16, gw))
    prefix = rng.choice([0, 0, 1])
    n, m = prefix + gh * gw, mh * mw
    # pairs x dims of a call: at most an eighth of the largest listed one (fp32 storage: a 64th, its kernels are slower)
    cap = 16 * 8 * 4096 * 256 * 128 // (8 if dtype == "bf16" else 64)
    heads = _log_int(rng, 1, max(1, min(384, cap // (n * max(m, 32) * d), (1 << 28) // (n * d))))
    H = rng.choice([h for h in (1, 2, 3, 5, 6, 8) if h <= heads])
    return _path(None, kind, heads // H, H, gh, gw, d, mh, mw, rng.randint(4, 12), prefix=prefix, dtype=dtype,
                 sigma=rng.choice([0.5, 1.0]))


def _n(case):
    return case["prefix"] + case["gh"] * case["gw"]


def _copy_regions(K, case, gen):
    """A tenth of the landmark regions of every head become copies of other regions (grids that the regions divide)."""
    B, H, _, d = K.shape
    mh, mw = case["mh"], case["mw"]
    m, rh, rw = mh * mw, case["gh"] // mh, case["gw"] // mw
    k = int(math.ceil(0.1 * m))
    perm = torch.rand((B, H, m), device=K.device, generator=gen).argsort(-1)
    g = K[:, :, case["prefix"]:].reshape(B, H, mh, rh, mw, rw, d).transpose(3, 4).reshape(B, H, m, rh * rw * d)
    idx = lambda p: p[..., None].expand(-1, -1, -1, g.shape[-1])
    g.scatter_(2, idx(perm[..., :k]), g.gather(2, idx(perm[..., k:2 * k])))
    K[:, :, case["prefix"]:] = g.reshape(B, H, mh, mw, rh, rw, d).transpose(3, 4).reshape(B, H, -1, d)


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    normal = lambda *shape: torch.randn(shape, device=dev, generator=gen)
    if case["kind"] == "solver":
        L = normal(case["batch"], case["m"], case["d"]) * 0.25          # pooled landmarks spread less than tokens
        W = torch.stack([torch.exp(-torch.cdist(x, x, p=1) / case["d"]) for x in L])
        return dict(case=case, W=W, dX=normal(*W.shape))
    if case["kind"] == "kernel":
        dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        A, Bm = (normal(case["batch"], k, case["d"]).to(dt) for k in (case["na"], case["nb"]))
        return dict(case=case, A=A, Bm=Bm, dK=normal(case["batch"], case["na"], case["nb"]))
    B, H, n, d, m = case["B"], case["H"], _n(case), case["d"], case["mh"] * case["mw"]
    f32 = case["dtype"] == "f32"
    dt = torch.float32 if f32 else torch.bfloat16
    Q, K, V, dO = (normal(B, H, n, d) * case["sigma"] for _ in range(4))
    if case["dup"]:
        _copy_regions(K, case, gen)
        V = torch.rand((B, H, n, d), device=dev, generator=gen) * 2 - 1
    st = dict(case=case, Q=Q.to(dt), K=K.to(dt), V=V.to(dt))
    var = torch.rand((H, m), device=dev, generator=gen) * 3e-3 + 1e-3
    p = binding.Problem(B, H, n, d, m, float(d), case["T"], ridge_eps=RIDGE, dtype=binding.LN_F32 if f32 else binding.LN_BF16,
                        whiten=torch.rsqrt(var + 1e-5), prefix=case["prefix"], gh=case["gh"], gw=case["gw"], mh=case["mh"],
                        mw=case["mw"])
    st["p"] = p
    buf = lambda size: torch.empty(size, dtype=torch.uint8, device=dev)
    if case["kind"] == "infer":
        st["ws"] = buf(ln.laplace_nystrom_workspace_bytes(p, False))
        return st
    st["dO"] = dO.to(dt)
    if case["kind"] == "block":
        st["blk"] = binding.Block(normal(H, d, 3, 3) * 0.2, rope_base=10000.0)
        # the two buffers are allocated by the first forward call and kept by the program
        _, st["saved"], st["ws"] = binding.laplace_attention_block_fwd(p, st["blk"], st["Q"], st["K"], st["V"])
        return st
    st["saved"] = buf(ln.laplace_nystrom_saved_bytes(p))
    st["ws"] = buf(ln.laplace_nystrom_workspace_bytes(p, True))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solver":
        X, hist, _ = ln.ns_pinv(state["W"], case["T"], RIDGE, want_hist=True)
        return dict(X=X, dW=ln.ns_pinv_bwd(state["W"], case["T"], RIDGE, 0.0, state["dX"], X_hist=hist))
    if kind == "kernel":
        lam = float(case["d"])
        Kmat = ln.l1_kernel(state["A"], state["Bm"], lam)
        dA, dB = ln.l1_kernel_bwd(state["A"], state["Bm"], lam, state["dK"], Kmat=Kmat)
        return dict(K=Kmat, dA=dA, dB=dB)
    p, Q, K, V = state["p"], state["Q"], state["K"], state["V"]
    if kind == "infer":
        return ln.laplace_nystrom_fwd(p, Q, K, V, ws=state["ws"])
    if kind == "block":
        O, saved, ws = binding.laplace_attention_block_fwd(p, state["blk"], Q, K, V, saved=state["saved"], ws=state["ws"])
        dQ, dK, dV, dW = binding.laplace_attention_block_bwd(p, state["blk"], Q, K, V, state["dO"], saved, ws)
        return dict(O=O, dQ=dQ, dK=dK, dV=dV, dW=dW)
    O = ln.laplace_nystrom_fwd(p, Q, K, V, saved=state["saved"], ws=state["ws"])
    dQ, dK, dV, _ = ln.laplace_nystrom_bwd(p, Q, K, V, state["dO"], state["saved"], ws=state["ws"])
    return dict(O=O, dQ=dQ, dK=dK, dV=dV)


def work(case):
    """Inputs once, outputs once; 2 (forward) and 3 (backward) operations per pair of rows and dim of a kernel block, and
    the matrix products of the path."""
    if case["kind"] == "solver":
        b, m, T = case["batch"], case["m"], case["T"]
        return {"bytes": 4 * b * 4 * m * m, "flops": b * T * (4 + 10) * m ** 3}
    if case["kind"] == "kernel":
        b, na, nb, d = (case[k] for k in ("batch", "na", "nb", "d"))
        e = 4 if case["dtype"] == "f32" else 2
        return {"bytes": b * (2 * (na + nb) * d * e + 2 * na * nb * 4), "flops": 5 * b * na * nb * d}
    n, m, d, heads, T = _n(case), case["mh"] * case["mw"], case["d"], case["B"] * case["H"], case["T"]
    e = 4 if case["dtype"] == "f32" else 2
    pairs = (2 * n * m + m * m) * d
    fwd = 2 * pairs + 4 * n * m * d + 4 * T * m ** 3 + 2 * m * m * d
    bwd = 3 * pairs + 8 * n * m * d + 10 * T * m ** 3 + 4 * m * m * d
    if case["kind"] == "infer":
        return {"bytes": heads * 4 * n * d * e, "flops": heads * fwd}
    extra = heads * n * d * (3 * 18 + 4 * 3) if case["kind"] == "block" else 0    # nine taps three times, four rotations
    return {"bytes": heads * 8 * n * d * e, "flops": heads * (fwd + bwd) + extra}


def tolerance(case):
    """About four times the error measured against float64 (the largest of the outputs, listed and drawn sizes)."""
    if case.get("dtype") == "bf16":
        return {"rel": 7e-3}                        # 1.7e-3: the rounding of the bf16 outputs
    if case["kind"] == "solver":
        return {"rel": 5e-5}                        # X_T 7e-6 at 228 landmarks, dW below 1e-6
    if case["kind"] == "kernel":
        return {"rel": 1e-5}                        # sums of up to 3000 terms in fp32
    if case["kind"] == "infer":
        return {"rel": 3e-5}                        # 6e-6 at 72 landmarks
    return {"rel": 2e-4}                            # dV 3e-5 at 49 landmarks, growing with their number
