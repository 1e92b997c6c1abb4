"""Cases that time this library's public entry points as a user's program calls them.

Sizes and data follow the repository's own workloads (``paper_1407_1785_gb300/synth.py``,
``bench.py`` and the tests): low-tubal-rank tensors, panning-texture videos and entrywise or
tube-wise corruptions, drawn here with torch on the GPU.  The ADMM solves run fewer iterations
than the benchmark's 100 to 200 so that a pass stays well under a second; threshold, rank and
conditioning still move through the regimes of such a solve, since the penalty grows by 10% an
iteration.  Tensors are flat FP32 buffers in column-major order.
"""
from __future__ import annotations

import math
import os
import random
from concurrent.futures import ThreadPoolExecutor

import torch

from paper_1407_1785_gb300 import libtsvd

FP32, XTF32 = libtsvd.PRECISION_FP32, libtsvd.PRECISION_3XTF32


# ------------------------------------------------------------------------------------ cases
# Keys of a case: op, n1, n2, n3[, n4] (modes), prec (arithmetic of the slice SVTs), then per
# op: rank of the low-rank part, p (observed fraction) or frac (corrupted fraction), iters.
def listed():
    return [
        # one proximal step on a small tensor: the cost of a call (launches, the wait, the reply)
        dict(name="prox_32x32x16", op="prox", n1=32, n2=32, n3=16, rank=3, prec=FP32),
        # de-noising one odd-sized 4-way tensor: modes 3 and 4 are transformed, ragged everywhere
        dict(name="prox_4way_61x75x3x21", op="prox", n1=61, n2=75, n3=3, n4=21, rank=5, prec=FP32),
        # the smallest solve: a low-rank tensor, half of it observed, 100 iterations
        dict(name="complete_32x32x16", op="complete", n1=32, n2=32, n3=16, rank=3, p=0.5,
             iters=100, prec=FP32),
        # grey video in-painting from 20% of its pixels, plain FP32
        dict(name="video_144x176x100", op="video", n1=144, n2=176, n3=100, p=0.2, iters=60,
             prec=FP32),
        # robust PCA with 10% gross errors, plain FP32: large slices of low rank
        dict(name="rpca_240x320x60", op="rpca", n1=240, n2=320, n3=60, rank=10, frac=0.1,
             iters=40, prec=FP32),
        # robust PCA of a video with noisy pixel tubes (group shrinkage), plain FP32
        dict(name="rpca_tube_144x256x80", op="rpca_tube", n1=144, n2=256, n3=80, frac=0.1,
             iters=40, prec=FP32),
        # an uneven batch, completions and robust PCA mixed, in one call: plain ...
        dict(name="batch_16", op="batch", count=16, shapes=1, iters=25, prec=FP32),
        # ... and in the mixed form (randomized sketches, split TF32 products)
        dict(name="batch_16_3xtf32", op="batch", count=16, shapes=1, iters=25, prec=XTF32),
        # 4-way colour video in-painting from 15% of its pixels, mixed form: the largest tensor
        dict(name="colour_288x352x3x60_3xtf32", op="video", n1=288, n2=352, n3=3, n4=60, p=0.15,
             iters=30, prec=XTF32),
        # the same robust PCA in the mixed form
        dict(name="rpca_240x320x60_3xtf32", op="rpca", n1=240, n2=320, n3=60, rank=10, frac=0.1,
             iters=60, prec=XTF32),
        # t-SVD compression of a surveillance-sized video to an eighth of its entries
        dict(name="compress_130x160x50", op="compress", n1=130, n2=160, n3=50, ratio=8.0,
             prec=FP32),
        # t-product of two tensors (a basis times its coefficients), split TF32 products
        dict(name="tproduct_144x176x100x50_3xtf32", op="tproduct", n1=144, n2=176, n3=100, n=50,
             prec=XTF32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same operations: slices 24 to 288 wide, tubes 5 to 100 long, 3- and 4-way."""
    most = max(_gvl(c) for c in listed() if c["op"] == "rpca" and c["prec"] == FP32)
    while True:
        op = rng.choice(["prox", "prox", "complete", "video", "rpca", "rpca", "rpca_tube", "batch",
                         "batch", "compress", "tproduct"])
        prec = FP32 if op in ("compress", "prox") else rng.choice([FP32, FP32, XTF32])
        c = dict(op=op, prec=prec)
        if op == "batch":
            c.update(count=rng.randint(3, 16), shapes=rng.randint(2, 10 ** 6),
                     iters=rng.randint(10, 25))
            return c
        n1, n2, n3 = _log_int(rng, 24, 288), _log_int(rng, 24, 288), _log_int(rng, 5, 100)
        if prec != FP32 and min(n1, n2) < 64:
            continue   # the mixed form is for slices a sketch is narrower than
        c.update(n1=n1, n2=n2, n3=n3)
        if rng.random() < 0.3 and op in ("prox", "video", "complete", "rpca") and n3 > 8:
            c.update(n3=3, n4=max(3, n3 // 2))
        if op in ("prox", "complete", "rpca"):
            c["rank"] = rng.randint(2, max(2, min(12, min(n1, n2) // 8)))
        if op in ("complete", "video"):
            c["p"] = round(rng.uniform(0.2, 0.6), 3)
        if op in ("rpca", "rpca_tube"):
            c["frac"] = round(rng.uniform(0.05, 0.15), 3)
        if op in ("complete", "video", "rpca", "rpca_tube"):
            c["iters"] = rng.randint(20, 60)
        if op == "compress":
            c["ratio"] = round(rng.uniform(2.0, 20.0), 2)
        if op == "tproduct":
            c["n"] = rng.randint(8, 96)
        if op == "tproduct" or _gvl(c) <= most:
            return c


# ----------------------------------------------------------------------------------- inputs
def _dims(c):
    return tuple(c[k] for k in ("n1", "n2", "n3", "n4") if k in c)


def _flat(t):
    """Column-major flat copy of an (n1, n2, ...) tensor."""
    return t.permute(*reversed(range(t.dim()))).contiguous().reshape(-1)


def _modes(dims):
    return tuple(range(2, len(dims)))


def _lowrank(dims, rank, g):
    """A * B (t-product over every mode from 3 on) of N(0, 1) factors, in FP64."""
    a = torch.randn((dims[0], rank) + dims[2:], generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn((rank, dims[1]) + dims[2:], generator=g, device="cuda", dtype=torch.float64)
    m = _modes(dims)
    c = torch.einsum("ir...,rj...->ij...", torch.fft.fftn(a, dim=m), torch.fft.fftn(b, dim=m))
    return torch.fft.ifftn(c, dim=m).real


def _texture_video(n1, n2, nt, g, bumps=20, dr=0.7, dc=0.4, noise=0.01):
    """A sum of Gaussian bumps panning by (0.7, 0.4) pixels a frame, bilinear, plus noise."""
    h, w = n1 + math.ceil(dr * nt) + 2, n2 + math.ceil(dc * nt) + 2
    par = torch.rand((bumps, 4), generator=g, device="cuda", dtype=torch.float64)
    yy = torch.arange(h, device="cuda", dtype=torch.float64)[:, None]
    xx = torch.arange(w, device="cuda", dtype=torch.float64)[None, :]
    tex = torch.zeros((h, w), device="cuda", dtype=torch.float64)
    for b in range(bumps):
        cy, cx, s, amp = par[b, 0] * h, par[b, 1] * w, 4 + 12 * par[b, 2], 0.2 + 0.8 * par[b, 3]
        tex += amp * torch.exp(-((yy - cy) ** 2 + (xx - cx) ** 2) / (2 * s * s))
    tex = (tex - tex.min()) / (tex.max() - tex.min())
    out = torch.empty((n1, n2, nt), device="cuda", dtype=torch.float64)
    for t in range(nt):
        y0, x0 = int(dr * t), int(dc * t)
        fy, fx = dr * t - y0, dc * t - x0
        out[:, :, t] = ((1 - fy) * (1 - fx) * tex[y0:y0 + n1, x0:x0 + n2]
                        + (1 - fy) * fx * tex[y0:y0 + n1, x0 + 1:x0 + 1 + n2]
                        + fy * (1 - fx) * tex[y0 + 1:y0 + 1 + n1, x0:x0 + n2]
                        + fy * fx * tex[y0 + 1:y0 + 1 + n1, x0 + 1:x0 + 1 + n2])
    return out + noise * torch.randn(out.shape, generator=g, device="cuda", dtype=torch.float64)


def _video(dims, g):
    if len(dims) == 3:
        return _texture_video(*dims, g)
    return torch.stack([_texture_video(dims[0], dims[1], dims[3], g) for _ in range(dims[2])], dim=2)


def _mask(dims, p, g):
    return (torch.rand(dims, generator=g, device="cuda") < p).to(torch.uint8)


def _gross_errors(dims, frac, g):
    hit = torch.rand(dims, generator=g, device="cuda") < frac
    return hit * (10 * torch.rand(dims, generator=g, device="cuda", dtype=torch.float64) - 5)


def _tube_errors(dims, frac, g, block=10):
    """Noisy pixels that stay the same within each block of frames."""
    n1, n2, n3 = dims
    hit = torch.rand((n1, n2, -(-n3 // block)), generator=g, device="cuda") < frac
    hit = hit.repeat_interleave(block, dim=2)[:, :, :n3]
    return hit * torch.randn(dims, generator=g, device="cuda", dtype=torch.float64)


def _batch_shapes(case):
    """Uneven shapes: n1, n2 in [48, 256], n3 in [8, 64], rank in [2, 12]; every other tensor is
    a completion (20 to 60% observed), the others robust PCA (5 to 15% corrupted)."""
    r = random.Random(case["shapes"])
    out = []
    for b in range(case["count"]):
        s = dict(op="rpca" if b % 2 else "complete", n1=r.randint(48, 256), n2=r.randint(48, 256),
                 n3=r.randint(8, 64), rank=r.randint(2, 12))
        s.update(frac=r.uniform(0.05, 0.15)) if b % 2 else s.update(p=r.uniform(0.2, 0.6))
        out.append(s)
    return out


def _lambda(case):
    if case["op"] == "rpca_tube":
        return 1.0 / math.sqrt(max(case["n1"], case["n2"]))
    return 1.0 / math.sqrt(max(case["n1"], case["n2"]) * math.prod(_dims(case)[2:]))


def _data(case, g):
    """The FP32 inputs of one tensor, as (n1, n2, ...) tensors: data, and the mask or None."""
    op, dims = case["op"], _dims(case)
    if op in ("complete", "video"):
        x = _video(dims, g) if op == "video" else _lowrank(dims, case["rank"], g)
        om = _mask(dims, case["p"], g)
        return (x * om).float(), om
    if op == "rpca":
        return (_lowrank(dims, case["rank"], g) + _gross_errors(dims, case["frac"], g)).float(), None
    if op == "rpca_tube":
        return (_video(dims, g) + _tube_errors(dims, case["frac"], g)).float(), None
    if op == "prox":   # a low-rank signal of unit entries in noise of a third of its size
        x = _lowrank(dims, case["rank"], g)
        x = x / x.std()
        return (x + torch.randn(dims, generator=g, device="cuda", dtype=torch.float64) / 3).float(), None
    if op == "compress":
        return _video(dims, g).float(), None
    raise ValueError(op)


def _tau(case):
    """Threshold at the noise's largest singular value in the Fourier slices."""
    dims = _dims(case)
    return math.sqrt(math.prod(dims[2:])) * (math.sqrt(dims[0]) + math.sqrt(dims[1])) / 3


def _kept(case):
    """Singular values that fit the compression ratio n1 n2 P / (kept (n1 + n2 + 1))."""
    n1, n2, p = case["n1"], case["n2"], math.prod(_dims(case)[2:])
    return max(1, int(n1 * n2 * p / (case["ratio"] * (n1 + n2 + 1))))


def _tproduct_dims(case):
    return (case["n1"], case["n2"], case["n3"]), (case["n2"], case["n"], case["n3"])


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    ctx = libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream,
                          precision=case["prec"],
                          sparse_mode=libtsvd.SPARSE_TUBE if case["op"] == "rpca_tube"
                          else libtsvd.SPARSE_ENTRY)
    st = dict(case=case, ctx=ctx)
    if case["op"] == "batch":
        st["problems"] = []
        for s in _batch_shapes(case):
            m, om = _data(s, g)
            q = dict(kind=s["op"], dims=_dims(s), M=_flat(m))
            if om is None:
                q["lam"] = _lambda(s)
            else:
                q["omega"] = _flat(om)
            q["out0"], q["out1"] = torch.empty_like(q["M"]), torch.empty_like(q["M"])
            st["problems"].append(q)
    elif case["op"] == "tproduct":
        da, db = _tproduct_dims(case)
        st["A"] = torch.randn(math.prod(da), generator=g, device="cuda")
        st["B"] = torch.randn(math.prod(db), generator=g, device="cuda")
        st["C"] = torch.empty(case["n1"] * case["n"] * case["n3"], device="cuda")
    else:
        m, om = _data(case, g)
        st["M"], st["omega"] = _flat(m), None if om is None else _flat(om)
        st["out0"], st["out1"] = torch.empty_like(st["M"]), torch.empty_like(st["M"])
    return st


# -------------------------------------------------------------------------------------- run
def run(state):
    case, ctx = state["case"], state["ctx"]
    op = case["op"]
    if op == "batch":
        ctx.solve_batched(state["problems"], case["iters"])
        return [(q["out0"], q["out1"]) for q in state["problems"]]
    if op == "tproduct":
        ctx.tproduct(state["A"], state["B"], state["C"], _tproduct_dims(case)[0], case["n"])
        return state["C"]
    dims, m, out0, out1 = _dims(case), state["M"], state["out0"], state["out1"]
    if op == "prox":
        ctx.tsvt(m, out0, dims, _tau(case))
        return out0
    if op == "compress":
        kept, _ = ctx.compress(m, dims, libtsvd.COMPRESS_GLOBAL, _kept(case), out0)
        return out0, kept
    if op in ("complete", "video"):
        ctx.tnn_complete(m, state["omega"], dims, case["iters"], out0, out1)
    else:
        ctx.trpca(m, dims, _lambda(case), case["iters"], out0, out1)
    return out0, out1


# ------------------------------------------------------------------------------------- work
def _distinct(dims):
    """Fourier slices that are not another one's conjugate."""
    return (math.prod(dims[2:]) + math.prod(2 - d % 2 for d in dims[2:])) // 2


def _gvl(case):
    """Flops of the slice SVDs: 4 (4 m n^2 + 8 n^3) per distinct slice and iteration (Golub and
    Van Loan's count, complex, singular values and right vectors)."""
    if case["op"] == "batch":
        return sum(_gvl(dict(s, iters=case["iters"])) for s in _batch_shapes(case))
    n, m = sorted((case["n1"], case["n2"]))
    return case.get("iters", 1) * _distinct(_dims(case)) * 4.0 * (4.0 * m * n * n + 8.0 * n ** 3)


def work(case):
    if case["op"] == "batch":
        each = [work(dict(s, iters=case["iters"], prec=case["prec"])) for s in _batch_shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    dims = _dims(case)
    n, p = math.prod(dims), math.prod(dims[2:])
    fft = 2.5 * math.log2(p)   # flops per real entry and transform
    if case["op"] == "tproduct":
        da, db = _tproduct_dims(case)
        na, nb, nc = math.prod(da), math.prod(db), case["n1"] * case["n"] * case["n3"]
        return {"bytes": 4.0 * (na + nb + nc),
                "flops": fft * (na + nb + nc) + 8.0 * case["n1"] * case["n2"] * case["n"] * _distinct(dims)}
    iters = case.get("iters", 1)
    flops = 2 * fft * n * iters
    if case["prec"] == FP32:
        flops += _gvl(case)
    else:   # three products with a sketch of the slice's rank (a video's is about a third of its width)
        k = case.get("rank", min(dims[:2]) // 3)
        flops += iters * _distinct(dims) * 24.0 * dims[0] * dims[1] * k
    each = {"prox": 8, "compress": 8, "complete": 13, "video": 13}.get(case["op"], 12)
    return {"bytes": float(each * n), "flops": flops}


# ------------------------------------------------------------------- the same in 64 bits
def _shrink_slice(b, tau):
    """D_tau of one slice through the eigenvectors of its smaller Gram matrix."""
    tall = b.shape[0] >= b.shape[1]
    lam, v = torch.linalg.eigh(b.mH @ b if tall else b @ b.mH)
    sig = lam.clamp_min(0).sqrt()
    keep = sig > tau
    v, f = v[:, keep], 1 - tau / sig[keep]
    return ((b @ v) * f) @ v.mH if tall else (v * f) @ (v.mH @ b)


def _half(dims):
    """Indices of the Fourier slices to compute, and of each one's conjugate partner."""
    idx = torch.arange(math.prod(dims[2:])).reshape(dims[2:])
    neg = idx
    for m in range(idx.dim()):
        neg = torch.roll(torch.flip(neg, (m,)), 1, m)
    idx, neg = idx.reshape(-1), neg.reshape(-1)
    own = idx <= neg
    return idx[own].tolist(), neg[own].tolist()


def _prox(y, tau, pool):
    dims, m = tuple(y.shape), _modes(y.shape)
    h = torch.fft.fftn(y, dim=m).reshape(dims[0], dims[1], -1).permute(2, 0, 1).contiguous()
    own, partner = _half(dims)
    for k, q, z in zip(own, partner, pool.map(lambda k: _shrink_slice(h[k], tau), own)):
        h[k] = z
        if q != k:
            h[q] = z.conj()
    return torch.fft.ifftn(h.permute(1, 2, 0).reshape(dims), dim=m).real


def _solve(case, m, om, pool):
    m = m.double().cpu()
    rho = 1e-2
    a = torch.zeros_like(m)   # Z or S
    d = torch.zeros_like(m)   # the scaled dual
    for _ in range(case["iters"]):
        nxt = min(1.1 * rho, 1e10)
        if om is not None:
            x = torch.where(om, m, a - d)
            a = _prox(x + d, 1 / rho, pool)
            d = (d + x - a) * (rho / nxt)
        else:
            x = _prox(m - a - d, 1 / rho, pool)
            r, k = m - d - x, _lambda(case) / rho
            if case["op"] == "rpca_tube":
                nrm = r.square().sum(dim=_modes(r.shape), keepdim=True).sqrt()
                a = torch.where(nrm > k, 1 - k / nrm, torch.zeros_like(nrm)) * r
            else:
                a = r.sign() * (r.abs() - k).clamp_min(0)
            d = (d + x + a - m) * (rho / nxt)
        rho = nxt
    return _flat(x), _flat(a)


def exact(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    workers = min(16, os.cpu_count() or 1)
    with ThreadPoolExecutor(workers, initializer=torch.set_num_threads, initargs=(1,)) as pool:
        if case["op"] == "batch":
            out = []
            for s in _batch_shapes(case):
                m, om = _data(s, g)
                if om is not None and case["prec"] != FP32:
                    out.append((None, None))   # see below
                    continue
                out.append(_solve(dict(s, iters=case["iters"]), m,
                                  None if om is None else om.bool().cpu(), pool))
            return out
        # A completion of a random low-rank tensor in the mixed form is far from the 64-bit one
        # until its last iterations: early on the sketch cuts a spectrum with no gap.
        if case["op"] == "complete" and case["prec"] != FP32:
            return None
        if case["op"] == "tproduct":
            da, db = _tproduct_dims(case)
            a = torch.randn(math.prod(da), generator=g, device="cuda").double().reshape(da[::-1])
            b = torch.randn(math.prod(db), generator=g, device="cuda").double().reshape(db[::-1])
            ch = torch.fft.fft(b, dim=0) @ torch.fft.fft(a, dim=0)   # (n3, n4, n1): column-major
            return torch.fft.ifft(ch, dim=0).real.reshape(-1)
        m, om = _data(case, g)
        if case["op"] == "prox":
            return _flat(_prox(m.double().cpu(), _tau(case), pool))
        if case["op"] == "compress":
            dims = _dims(case)
            h = torch.fft.fftn(m.double().cpu(), dim=_modes(dims))
            h = h.reshape(dims[0], dims[1], -1).permute(2, 0, 1).contiguous()
            svd = list(pool.map(lambda k: torch.linalg.svd(h[k], full_matrices=False), range(h.shape[0])))
            least = torch.cat([s for _, s, _ in svd]).sort(descending=True)[0][_kept(case) - 1]
            kept = 0
            for k, (u, s, vh) in enumerate(svd):
                keep = s >= least * (1 - 1e-12)   # a conjugate slice's equal value goes with it
                kept += int(keep.sum())
                h[k] = (u[:, keep] * s[keep]) @ vh[keep]
            z = torch.fft.ifftn(h.permute(1, 2, 0).reshape(dims), dim=_modes(dims)).real
            return _flat(z), None
        return _solve(case, m, None if om is None else om.bool().cpu(), pool)
