"""The library's workloads as single calls through its Python entry points.

Each case is one call (or one training step) that a user's program makes:
Gram matrices and their RBF lift, pairs of uneven lengths, the MMD^2 loss with
its gradient, long pairs forward and backward, the solution surface, a small
gradient step, in FP32 and FP64.  ``listed`` holds fixed sizes, ``draw`` gives
further ones of the same ranges, ``prepare`` makes a case's inputs from a seed,
``run`` is one pass, ``work`` what a pass cannot do without, and ``exact`` the
same outputs from a plain torch FP64 solve that uses none of the library.

Paths are Brownian walks rescaled to O(1) amplitude (steps N(0, 1/(L d))),
with a time channel t in [0, 1] where the workload is time-augmented.
"""
from __future__ import annotations

import math

import torch

from paper_2006_14794_gb300 import sigk

DEVICE = "cuda"


def _case(kind, B, By, L, M, d, lam, dtype="f32", kernel="linear", scheme="explicit", time=True, **more):
    return dict(kind=kind, B=B, By=By, L=L, M=M, d=d, lam=lam, dtype=dtype, kernel=kernel, scheme=scheme,
                time=time, **more)


def listed():
    return [
        # the smallest call: a Gram of eight short paths in double precision (latency, launches)
        dict(_case("gram", 8, 8, 32, 32, 3, 1, dtype="f64"), name="gram_small_f64"),
        # a kernel-method Gram of 256 x 256 paths in single precision
        dict(_case("gram", 256, 256, 128, 128, 8, 2), name="gram_256"),
        # the same Gram with the RBF static kernel
        dict(_case("gram", 256, 256, 128, 128, 8, 2, kernel="rbf"), name="gram_256_rbf"),
        # a Gram in double precision, as a reference run of the FP32 one asks for it
        dict(_case("gram", 64, 64, 128, 128, 8, 2, dtype="f64"), name="gram_64_f64"),
        # a data set of time series of uneven lengths, packed
        dict(_case("varlen", 4096, 0, 16, 512, 16, 1, time=False), name="uneven_4096"),
        # a generative model's training step: MMD^2 and its gradient in the generated paths
        dict(_case("mmd", 128, 128, 256, 256, 32, 1, time=False), name="mmd_128"),
        # the same loss with the RBF static kernel
        dict(_case("mmd", 128, 128, 256, 256, 32, 1, kernel="rbf", time=False), name="mmd_128_rbf"),
        # the loss and its gradient in double precision, as a gradient check runs it
        dict(_case("mmd", 16, 16, 64, 64, 32, 1, dtype="f64", time=False), name="mmd_16_f64"),
        # few long series of many channels
        dict(_case("pairs", 64, 0, 4096, 4096, 64, 1), name="long_64"),
        # their gradient
        dict(_case("pairs_grad", 64, 0, 4096, 4096, 64, 1), name="long_64_grad"),
        # the whole solution on the sample grid (the surfaces that the paper plots and regresses on)
        dict(_case("surface", 16384, 0, 128, 128, 8, 2), name="surface_16384"),
        # a minibatch step of a model on short ragged series: a Gram with both gradients
        dict(_case("gram_grad", 24, 17, 50, 71, 5, 1), name="minibatch_grad"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(("gram", "gram", "gram", "varlen", "mmd", "mmd", "pairs", "pairs_grad", "surface",
                       "gram_grad"))
    dtype = "f64" if kind in ("gram", "mmd", "pairs") and rng.random() < 0.3 else "f32"
    f64 = dtype == "f64"
    kernel = "rbf" if kind in ("gram", "mmd") and rng.random() < 0.35 else "linear"
    scheme = "implicit" if kind == "gram" and rng.random() < 0.2 else "explicit"
    if kind == "gram":
        top = 64 if f64 else 256
        return _case(kind, _log_int(rng, 6, top), _log_int(rng, 6, top), _log_int(rng, 16, 200),
                     _log_int(rng, 16, 200), rng.randint(2, 16), rng.randint(0, 2), dtype, kernel, scheme)
    if kind == "varlen":
        lo = _log_int(rng, 8, 64)
        return _case(kind, _log_int(rng, 64, 4096), 0, lo, rng.randint(2 * lo, 512), rng.randint(2, 24),
                     rng.randint(0, 1), time=False)
    if kind == "mmd":
        top, long = (16, 64) if f64 else (128, 256)
        L = _log_int(rng, 16, long)
        return _case(kind, _log_int(rng, 6, top), _log_int(rng, 6, top), L, L, rng.randint(2, 40),
                     rng.randint(0, 1), dtype, kernel, time=False)
    if kind in ("pairs", "pairs_grad"):
        top = 1024 if f64 else 4096
        return _case(kind, _log_int(rng, 4, 16 if f64 else 64), 0, _log_int(rng, 300, top),
                     _log_int(rng, 300, top), rng.randint(4, 64), rng.randint(0, 1), dtype)
    if kind == "surface":
        return _case(kind, _log_int(rng, 64, 16384), 0, _log_int(rng, 16, 128), _log_int(rng, 16, 128),
                     rng.randint(2, 12), rng.randint(0, 2))
    return _case(kind, _log_int(rng, 6, 48), _log_int(rng, 6, 48), _log_int(rng, 16, 120),
                 _log_int(rng, 16, 120), rng.randint(2, 16), rng.randint(0, 1))


def draw(rng):
    """One more case of the listed ranges, no larger than the listed case of its kind and type."""
    most = {}
    for c in listed():
        key = (c["kind"], c["dtype"])
        most[key] = max(most.get(key, 0.0), work(c)["flops"])
    most[("pairs", "f64")] = most[("gram", "f64")]
    while True:
        c = _draw_once(rng)
        if work(c)["flops"] <= most[(c["kind"], c["dtype"])]:
            return c


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _variant(case):
    return sigk.Variant(scheme=case["scheme"], static_kernel=case["kernel"], sigma=1.0)


def _walks(gen, B, L, d, time):
    w = torch.randn(B, L, d, generator=gen, device=DEVICE, dtype=torch.float64) / math.sqrt(L * d)
    w[:, 0] = 0
    w = w.cumsum(1)
    if time:
        w[:, :, 0] = torch.arange(L, device=DEVICE, dtype=torch.float64) / max(L - 1, 1)
    return w


def _packed(gen, lengths, d):
    """Walks of the given lengths one after another, and their offsets [B + 1]."""
    off = torch.zeros(len(lengths) + 1, dtype=torch.int64)
    off[1:] = lengths.cumsum(0)
    per_row = torch.repeat_interleave(lengths, lengths).to(DEVICE, torch.float64)
    off = off.to(DEVICE)
    w = torch.randn(per_row.numel(), d, generator=gen, device=DEVICE, dtype=torch.float64)
    w /= (per_row * d).sqrt()[:, None]
    w[off[:-1]] = 0
    w = w.cumsum(0)
    w -= torch.repeat_interleave(w[off[:-1]], lengths.to(DEVICE), dim=0)
    return w, off


def _lengths(case, seed):
    """The uneven lengths of a case: host integers, so that every user of the seed has the same."""
    gen = torch.Generator().manual_seed(seed)
    lo, hi = case["L"], case["M"]
    return [torch.randint(lo, hi + 1, (case["B"],), generator=gen) for _ in range(2)]


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    kind, B, By, L, M, d = (case[k] for k in ("kind", "B", "By", "L", "M", "d"))
    s = dict(kind=kind, lam=case["lam"], variant=_variant(case))
    if kind == "varlen":
        Ls, Ms = _lengths(case, seed)
        X, s["x_off"] = _packed(gen, Ls, d)
        Y, s["y_off"] = _packed(gen, Ms, d)
        s["max_len"] = M
    else:
        X = _walks(gen, B, L, d, case["time"])
        Y = _walks(gen, B if kind in ("pairs", "pairs_grad", "surface") else By, M, d, case["time"])
    if kind == "mmd":   # the two samples differ by a drift of 0.57 in all over unit time
        Y += 0.1 * math.sqrt(32 / d) * (torch.arange(M, device=DEVICE) / (M - 1))[None, :, None]
    s["X"], s["Y"] = X.to(_dtype(case)), Y.to(_dtype(case))
    if kind in ("mmd", "pairs_grad", "gram_grad"):
        s["X"].requires_grad_(True)
    if kind in ("pairs_grad", "gram_grad"):
        s["Y"].requires_grad_(True)
        shape = (B,) if kind == "pairs_grad" else (B, By)
        s["g"] = torch.randn(shape, generator=gen, device=DEVICE, dtype=_dtype(case))
    return s


def run(s):
    X, Y, lam, variant = s["X"], s["Y"], s["lam"], s["variant"]
    kind = s["kind"]
    if kind == "gram":
        return sigk.gram(X, Y, lam, variant=variant)
    if kind == "pairs":
        return sigk.pairs(X, Y, lam, variant=variant)
    if kind == "varlen":
        return sigk.pairs_varlen(X, s["x_off"], Y, s["y_off"], lam, s["max_len"], variant=variant)
    if kind == "surface":
        return sigk.pairs_surface(X, Y, lam, variant=variant)
    if kind == "mmd":
        loss = sigk.mmd2_loss(X, Y, lam, variant=variant)
        (dX,) = torch.autograd.grad(loss, X)
        return loss.detach(), dX
    function = sigk.SigKernelPairs if kind == "pairs_grad" else sigk.SigKernelGram
    k = function.apply(X, Y, lam, variant)
    dX, dY = torch.autograd.grad(k, (X, Y), s["g"])
    return k.detach(), dX, dY


def work(case):
    """Inputs read once, outputs written once; 3 operations a refined cell for the scheme and 4 for
    its adjoint, 2 d a coarse cell for its increment product (RBF: for a point's kernel value) and
    2 d for each path's gradient."""
    kind, B, By, L, M, d, lam = (case[k] for k in ("kind", "B", "By", "L", "M", "d", "lam"))
    size = 8 if case["dtype"] == "f64" else 4
    if kind == "varlen":
        mean = (L + M) / 2
        cells, points, out = B * (mean - 1) ** 2, 2 * B * mean, B
    elif kind == "mmd":
        n = B * (B + 1) / 2 + By * (By + 1) / 2 + B * By
        cells, points, out = n * (L - 1) * (M - 1), B * L + By * M, 1
    elif kind in ("gram", "gram_grad"):
        cells, points, out = B * By * (L - 1) * (M - 1), B * L + By * M, B * By
    else:
        cells, points, out = B * (L - 1) * (M - 1), B * (L + M), B
    flops = cells * (3 * 4 ** lam + 2 * d)
    if kind == "surface":
        out += B * L * M
    elif kind == "mmd":   # the pairs that the gradient in X goes through
        flops += (B * (B + 1) / 2 + B * By) * (L - 1) * (M - 1) * (4 * 4 ** lam + 2 * d)
        out += B * L * d
    elif kind in ("pairs_grad", "gram_grad"):
        flops += cells * (4 * 4 ** lam + 4 * d)
        out += points * d
    return {"bytes": size * (points * d + out), "flops": flops}


# ---- the same outputs in plain torch, FP64 -----------------------------------


def _coefficients(x, y, kernel):
    """<dx_p, dy_q> of paired paths x [n, L, d], y [n, M, d], or the second difference of the RBF
    kernel (sigma = 1): [nx * ny, n], pairs innermost."""
    if kernel == "rbf":
        dist = (x * x).sum(2)[:, :, None] + (y * y).sum(2)[:, None, :] - 2 * x @ y.transpose(1, 2)
        k = torch.exp(-0.5 * dist)
        G = k[:, 1:, 1:] - k[:, :-1, 1:] - k[:, 1:, :-1] + k[:, :-1, :-1]
    else:
        G = x.diff(dim=1) @ y.diff(dim=1).transpose(1, 2)
    return G.reshape(G.shape[0], -1).t().contiguous()


def _solve(G, nx, ny, lam, scheme, gout=None, nodes=False):
    """The scheme on the refined grid, one anti-diagonal at a time, for n pairs at once.
    Returns k [n], dk/dG (scaled by gout [n]) where gout is given, and the values at the sample
    grid's nodes [n, nx + 1, ny + 1] where nodes is set."""
    S, n = 1 << lam, G.shape[1]
    Ni, Nj = nx << lam, ny << lam
    h = G / (2 * 4 ** lam)
    # k(i+1,j+1) = mult (k(i+1,j) + k(i,j+1)) - k(i,j) in either scheme
    mult = 1 + h if scheme == "explicit" else (1 + h / 2) / (1 - h / 2)
    rows = torch.arange(Ni + 1, device=G.device)

    def span(s):   # the nodes (i, s - i) off the boundary
        return max(1, s - Nj), min(Ni, s - 1) + 1

    def cells(s):
        lo, hi = span(s)
        i = rows[lo:hi]
        return ((i - 1) >> lam) * ny + ((s - i - 1) >> lam)

    surf = torch.ones(nx + 1, ny + 1, n, dtype=G.dtype, device=G.device) if nodes else None
    sums = []
    older = torch.ones(Ni + 1, n, dtype=G.dtype, device=G.device)
    old = torch.ones_like(older)
    for s in range(2, Ni + Nj + 1):
        lo, hi = span(s)
        both = old[lo:hi] + old[lo - 1:hi - 1]
        new = torch.ones_like(old)
        new[lo:hi] = mult[cells(s)] * both - older[lo - 1:hi - 1]
        if gout is not None:
            sums.append(both)
        if nodes and s % S == 0:
            i = rows[(lo + S - 1) // S * S:hi:S]
            surf[i >> lam, (s - i) >> lam] = new[i]
        older, old = old, new
    k = old[Ni]
    dG = None
    if gout is not None:
        dmult = torch.zeros_like(G)
        # a node's adjoint: A(i,j) = W(i,j+1) + W(i+1,j) - A(i+1,j+1), W = mult A
        A1 = torch.zeros(Ni + 2, n, dtype=G.dtype, device=G.device)   # diagonal s + 1
        A2, W1 = torch.zeros_like(A1), torch.zeros_like(A1)
        for s in range(Ni + Nj, 1, -1):
            lo, hi = span(s)
            A = torch.zeros_like(A1)
            A[lo:hi] = W1[lo:hi] + W1[lo + 1:hi + 1] - A2[lo + 1:hi + 1]
            if s == Ni + Nj:
                A[Ni] = gout
            at = cells(s)
            dmult.index_add_(0, at, A[lo:hi] * sums[s - 2])
            W1 = torch.zeros_like(A1)
            W1[lo:hi] = mult[at] * A[lo:hi]
            A1, A2 = A, A1
            sums[s - 2] = None
        dG = dmult * ((1 if scheme == "explicit" else 1 / (1 - h / 2) ** 2) / (2 * 4 ** lam))
    return k, dG, surf.permute(2, 0, 1) if nodes else None


def _pairwise(case, X, Y, ix, iy, gout=None, nodes=False):
    """k of the pairs (X[ix], Y[iy]); with gout the gradients are added into X.grad and Y.grad."""
    nx, ny = X.shape[1] - 1, Y.shape[1] - 1
    per_pair = nx * ny * (4 ** case["lam"] / 4 if gout is not None else 1)
    chunk = max(1, int(2 ** 30 / per_pair))
    ks, surfs = [], []
    for a in range(0, len(ix), chunk):
        i, j = ix[a:a + chunk], iy[a:a + chunk]
        with torch.set_grad_enabled(gout is not None):
            G = _coefficients(X[i], Y[j], case["kernel"])
        with torch.no_grad():
            k, dG, surf = _solve(G.detach(), nx, ny, case["lam"], case["scheme"],
                                 None if gout is None else gout[a:a + chunk], nodes)
        if gout is not None:
            G.backward(dG)
        ks.append(k)
        surfs.append(surf)
    return (torch.cat(ks), torch.cat(surfs)) if nodes else torch.cat(ks)


def _padded(P, off, L):
    """Packed paths as [B, L, d], each continued by its last point (zero increments leave k alone)."""
    first, count = off[:-1, None], off[1:, None] - off[:-1, None]
    at = torch.arange(L, device=P.device)[None, :]
    return P[first + torch.minimum(at, count - 1)]


def exact(case, seed):
    s = prepare(case, seed)
    kind, B, By = case["kind"], case["B"], case["By"]
    X, Y = (s[n].detach().double() for n in ("X", "Y"))
    if kind == "varlen":
        X, Y = _padded(X, s["x_off"], case["M"]), _padded(Y, s["y_off"], case["M"])
    one = torch.arange(B, device=DEVICE)
    if kind in ("pairs", "varlen"):
        return _pairwise(case, X, Y, one, one)
    if kind == "surface":
        return _pairwise(case, X, Y, one, one, nodes=True)
    if kind == "pairs_grad":
        ix, iy = one, one
    else:
        ix, iy = one.repeat_interleave(By), torch.arange(By, device=DEVICE).repeat(B)
    if kind == "gram":
        return _pairwise(case, X, Y, ix, iy).view(B, By)
    X.requires_grad_(True)
    Y.requires_grad_(True)
    if kind in ("pairs_grad", "gram_grad"):
        g = s["g"].double()
        k = _pairwise(case, X, Y, ix, iy, g.reshape(-1))
        return k.view(g.shape), X.grad, Y.grad
    # the unbiased MMD^2: means over i != j of k(x_i, x_j) and k(y_i, y_j), less twice the mean of k(x_i, y_j)
    jx = one.repeat(B)
    gxx = (one.repeat_interleave(B) != jx).double() / (B * (B - 1))
    kxx = _pairwise(case, X, X, one.repeat_interleave(B), jx, gxx)
    kxy = _pairwise(case, X, Y, ix, iy, torch.full((B * By,), -2.0 / (B * By), device=DEVICE, dtype=torch.float64))
    y1 = torch.arange(By, device=DEVICE)
    yi, yj = y1.repeat_interleave(By), y1.repeat(By)
    kyy = _pairwise(case, Y.detach(), Y.detach(), yi, yj)
    loss = (kxx * gxx).sum() + kyy[yi != yj].mean() - 2 * kxy.mean()
    return loss, X.grad
