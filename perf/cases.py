"""The work this framework is run for, as cases to be timed and compared: the saliency map of a seismic
volume (the paper's windows 8, 16 and 32, each precision), its adjoints layer by layer, one step of fitting
the combination to an interpreter's template, the 2-D section mode and the paper's adaptive weight filter.

A case is a dict of plain values.  Its "kind" is the entry point:
  forward   Saliency.saliency: volume -> map S, weights W, features E and per-dimension maps S3
  adjoint   sal_local_spectra_project_backward: feature gradients -> volume gradient
  fit       autograd.saliency: the map, the squared distance to the template, gradients of W and alpha
  dcs       sal_center_surround_backward: map gradients -> feature gradients and alpha gradients
  adapt     sal_adapt_weights: the paper's sequential filters over the maps and a template

Volumes are synthetic layered seismic (the paper's field surveys are not public): Ricker-convolved
reflectivity bent by folds and cut by faults, with noise of a tenth of its rms, all made on the GPU.
"""
import math

import numpy as np
import torch

import paper_2201_06174_gb300 as sal
from paper_2201_06174_gb300 import autograd as sal_autograd

R, SIGMA = 3, 1.5
VOLUME_DIRECTIONS = ((1, 0, 0), (0, 1, 0), (1, 1, 0))     # t, x, t-x: the default window
SECTION_DIRECTIONS = ((0, 1, 0), (0, 0, 1), (0, 1, 1))    # the same directions in the plane of a section


def _case(kind, T, X, Y, n=16, prec="fp32", feature="abs", boundary="symmetric", taper="rect", stride=1,
          weights="equal", section=False, method="", block=0, name=None):
    c = dict(kind=kind, T=T, X=X, Y=Y, n=n, prec=prec, feature=feature, boundary=boundary, taper=taper,
             stride=stride, weights=weights, section=section, method=method, block=block)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a thumbnail with a template, the size of the smoke test: what one call costs however little it computes
        _case("forward", 10, 9, 37, n=8, weights="template", name="thumbnail_fp32_n8"),
        # one step of fitting weights to a template on the smallest benchmark volume: many short launches
        _case("fit", 48, 48, 48, n=8, prec="bf16", weights="given", name="fit48_bf16_n8"),
        # the paper's pipeline on one ordinary volume, 16^3 cubes, in the fast and in the exact form
        _case("forward", 128, 128, 128, n=16, prec="bf16", name="salt128_bf16_n16"),
        _case("forward", 128, 128, 128, n=16, weights="template", name="salt128_fp32_n16"),
        # the same volumes' gradients, the larger part of a differentiated call
        _case("adjoint", 128, 128, 128, n=16, prec="bf16", name="adjoint128_bf16_n16"),
        _case("adjoint", 128, 128, 128, n=16, name="adjoint128_fp32_n16"),
        # one inline section, odd sides, as a plane
        _case("forward", 1, 462, 951, n=16, prec="bf16", weights="given", section=True, name="section_bf16_n16"),
        # a survey block with the smallest window: the stencil and the normalisation weigh most here
        _case("forward", 256, 384, 192, n=8, prec="fp16", name="block_fp16_n8"),
        # the largest window, on a cut of the same block in the fast form and on a smaller one in the exact form
        _case("forward", 64, 96, 96, n=32, prec="bf16", name="cut_bf16_n32"),
        _case("forward", 48, 64, 64, n=32, name="cut_fp32_n32"),
        # the full survey (rows of 651 samples): the gradient of its features
        _case("adjoint", 462, 951, 651, n=16, prec="bf16", name="survey_adjoint_bf16_n16"),
        # the paper's filter for all its results, one chain over a whole volume
        _case("adapt", 96, 96, 96, weights="template", method="nlms", name="nlms96"),
    ]


def _sides(rng, voxels, least=5):
    """Three sides of about `voxels` voxels in all, odd or even as they come, none much longer than the others."""
    side = voxels ** (1.0 / 3.0)
    a, b = (math.exp(rng.uniform(-0.6, 0.6)) for _ in range(2))
    return tuple(max(least, int(round(v))) for v in (side * a, side * b, side / (a * b)))


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("forward", "forward", "forward", "adjoint", "adjoint", "fit", "dcs", "section", "adapt"))
    prec = rng.choice(("fp32", "bf16", "fp16"))
    boundary = rng.choice(("symmetric", "symmetric", "symmetric", "periodic", "zero"))
    feature = rng.choice(("abs", "abs", "abs", "energy"))
    taper = rng.choice(("rect", "rect", "rect", "hann"))
    weights = rng.choice(("equal", "given", "template"))
    if kind == "forward":
        n = rng.choice((8, 16, 16, 32))
        most = {8: 2e7, 16: 2e7 if prec != "fp32" else 4e6, 32: 1e6 if prec != "fp32" else 2.5e5}[n]
        T, X, Y = _sides(rng, _spread(rng, 3e3, most))
        stride = rng.choice((1, 1, 1, 2, 3))
        return _case(kind, T, X, Y, n, prec, feature, boundary, taper, stride, weights)
    if kind == "section":
        v = _spread(rng, 3e3, 2e6)
        a = math.exp(rng.uniform(-0.6, 0.6))
        X, Y = (max(16, int(round(s))) for s in (math.sqrt(v) * a, math.sqrt(v) / a))
        return _case("forward", 1, X, Y, rng.choice((8, 16)), prec, "abs", "symmetric", "rect", 1, "given", True)
    if kind == "adjoint":
        n = rng.choice((8, 16, 16))
        T, X, Y = _sides(rng, _spread(rng, 3e3, 2e7 if prec != "fp32" else 3e6))
        return _case(kind, T, X, Y, n, prec, feature, boundary, taper)
    if kind == "fit":
        n = rng.choice((8, 16))
        T, X, Y = _sides(rng, _spread(rng, 3e3, 4e6))
        return _case(kind, T, X, Y, n, prec, "abs", boundary, "rect", 1, "given")
    if kind == "dcs":
        T, X, Y = _sides(rng, _spread(rng, 3e3, 3e7))
        return _case(kind, T, X, Y, 8, "fp32", boundary=boundary)
    T, X, Y = _sides(rng, _spread(rng, 3e3, 9e5))
    return _case("adapt", T, X, Y, boundary=boundary, weights="template", method=rng.choice(("lms", "nlms", "nlms", "rls")),
                 block=rng.choice((0, 0, 4, 7)))


# ---- inputs -------------------------------------------------------------------------------------

def _volume(case, seed):
    """(V, D): a layered volume and the template of its faults, float32 on the GPU."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed))
    r = np.random.RandomState(int(seed) % (1 << 32))
    T, X, Y = case["T"], case["X"], case["Y"]
    pad = 40
    length = T + 2 * pad
    # reflection coefficients at layer tops 2 to 6 samples apart, convolved with a 30 Hz Ricker at 4 ms
    tops = np.cumsum(r.randint(2, 7, length))
    coeff = np.zeros(length)
    coeff[tops[tops < length]] = r.randn(int((tops < length).sum()))
    tau = (np.arange(-12, 13) * 0.004 * 30.0 * math.pi) ** 2
    trace = torch.from_numpy(np.convolve(coeff, (1 - 2 * tau) * np.exp(-tau), "same").astype(np.float32)).to(dev)
    x = torch.arange(X, device=dev, dtype=torch.float32)[:, None]
    y = torch.arange(Y, device=dev, dtype=torch.float32)[None, :]
    fold = 5.0 * torch.sin(x * (2 * math.pi / 64) + float(r.rand()) * 6) * torch.sin(y * (2 * math.pi / 64))
    faults = []
    for _ in range(3):
        strike, dip = r.rand() * 2 * math.pi, math.radians(50 + 25 * r.rand())
        cx, cy = X * (0.25 + 0.5 * r.rand()), Y * (0.25 + 0.5 * r.rand())
        along = (x - cx) * math.sin(strike) + (y - cy) * math.cos(strike)
        faults.append((along * math.sin(dip), math.cos(dip), T * r.rand(), 2.0 + 6.0 * r.rand()))
    V = torch.empty((T, X, Y), device=dev)
    D = torch.zeros((T, X, Y), device=dev)
    for t in range(T):
        z = t + pad + fold
        for side, ct, t0, throw in faults:
            d = side + ct * (t - t0)
            z = z - throw * (d > 0)
            D[t].masked_fill_(d.abs() < 1.0, 1.0)
        z = z.clamp(0, length - 1.001)
        i = z.floor()
        f = z - i
        i = i.long()
        V[t] = trace[i] * (1 - f) + trace[i + 1] * f
    V += torch.randn(V.shape, generator=g, device=dev) * (0.1 * float(V.square().mean().sqrt()) + 1e-3)
    return V, D


def _maps(case, seed):
    """(S3, D): three positive maps that stand out at faults, as center-surround maps do, and for a desired map the
    first of them with some noise (the paper adapts to one of the maps; a mask of zeros would let W die out)."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed))
    shape = (case["T"], case["X"], case["Y"])
    _, mask = _volume(case, seed)
    S3 = torch.empty((3,) + shape, device=dev)
    for m in range(3):
        S3[m] = torch.randn(shape, generator=g, device=dev).abs() * 0.1 + mask * (0.5 - 0.1 * m) * torch.rand(
            shape, generator=g, device=dev) + 0.05
    return S3, S3[0] / S3[0].max() + 0.05 * torch.randn(shape, generator=g, device=dev)


def _engine(case):
    p = sal.Params(n=case["n"], prec=case["prec"], feature=case["feature"], boundary=case["boundary"],
                   taper=case["taper"], stride=case["stride"], R=R, sigma=SIGMA,
                   directions=SECTION_DIRECTIONS if case["section"] else VOLUME_DIRECTIONS)
    return sal.Saliency((case["T"], case["X"], case["Y"]), p)


def _weights(case):
    return (0.0, 0.5, 0.5) if case["section"] else (0.5, 0.3, 0.2)


def _gradient(case, seed, planes):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7919)
    shape = (planes, case["T"], case["X"], case["Y"])
    return torch.randn(shape, generator=g, device="cuda")


def prepare(case, seed):
    st = {"case": case, "engine": _engine(case)}
    kind = case["kind"]
    if kind == "adapt":
        st["S3"], st["D"] = _maps(case, seed)
        blocks = -(-case["Y"] // case["block"]) if case["block"] else 1
        st["W"] = torch.empty((blocks, 3), device="cuda")
        st["err2"] = torch.empty(case["T"] * case["X"] * case["Y"], device="cuda")
        return st
    if kind == "dcs":
        st["E"] = _maps(case, seed)[0]
        st["gS3"] = _gradient(case, seed, 3)
        st["gE"] = torch.empty_like(st["E"])
        st["galpha"] = torch.empty(3, device="cuda")
        return st
    V, D = _volume(case, seed)
    st["V"] = V
    if kind == "adjoint":
        st["gE"] = _gradient(case, seed, 3)
        st["gV"] = torch.empty_like(V)
    elif kind == "fit":
        st["D"] = D
        st["W"] = torch.tensor(_weights(case), device="cuda", requires_grad=True)
        st["alpha"] = torch.tensor((1.0, 0.9, 1.1), device="cuda", requires_grad=True)
    else:
        st["D"] = D if case["weights"] == "template" else None
        st["W"] = torch.tensor(_weights(case), device="cuda") if case["weights"] == "given" else None
    return st


def run(st):
    kind, eng = st["case"]["kind"], st["engine"]
    if kind == "forward":
        return eng.saliency(st["V"], D=st["D"], W=st["W"], intermediates=True)
    if kind == "adjoint":
        sal.sal_local_spectra_project_backward(eng.h, st["V"], st["gE"], st["gV"])
        return {"gV": st["gV"]}
    if kind == "fit":
        S = sal_autograd.saliency(st["V"], st["W"], st["alpha"], eng)
        loss = 0.5 * (S - st["D"]).square().mean()
        gW, galpha = torch.autograd.grad(loss, (st["W"], st["alpha"]))
        return {"S": S.detach(), "loss": loss.detach(), "gW": gW, "galpha": galpha}
    if kind == "dcs":
        sal.sal_center_surround_backward(eng.h, st["E"], st["gS3"], st["gE"], st["galpha"])
        return {"gE": st["gE"], "galpha": st["galpha"]}
    sal.sal_adapt_weights(eng.h, st["S3"], st["D"], st["W"], method=st["case"]["method"], sections=st["case"]["block"],
                          err2=st["err2"])
    return {"W": st["W"], "err2": st["err2"]}


def work(case):
    """Bytes: inputs read and outputs written once.  Flops: per bin of the half spectrum one complex multiply-add
    (a sliding DFT's update, 8), the magnitude (4) and three weighted sums (6); the adjoint takes the update, the
    magnitude, the weight (5), the direction (3) and the inverse's update (8).  18 neighbours of 3 maps."""
    N, n = case["T"] * case["X"] * case["Y"], case["n"]
    cubes = N if case["stride"] == 1 else -(-case["T"] // case["stride"]) * -(-case["X"] // case["stride"]) * -(
        -case["Y"] // case["stride"])
    bins = (n // 2 + 1) * n * (1 if case["section"] else n)
    if case["section"]:
        cubes, bins = N, (n // 2 + 1) * n
    kind, D = case["kind"], 4 * N * (case["weights"] == "template")
    if kind == "forward":
        return {"bytes": 4 * N * 8 + D, "flops": cubes * bins * 18 + N * 3 * 18 * 4}
    if kind == "adjoint":
        return {"bytes": 4 * N * 5, "flops": cubes * bins * 28}
    if kind == "fit":
        return {"bytes": 4 * N * 3, "flops": cubes * bins * 18 + N * 3 * 18 * 12}
    if kind == "dcs":
        return {"bytes": 4 * N * 9, "flops": N * 3 * 18 * 11}
    return {"bytes": 4 * N * 5, "flops": N * (60 if case["method"] == "rls" else 20)}


# ---- the same in 64 bits, plain torch -----------------------------------------------------------

F8 = torch.float64
WINDOW_COST = 4e10   # windows x window size above which no 64-bit value is given


def _ext(i, n, mode):
    """Source sample of each extended index of one axis; -1 outside a zero-extended volume."""
    if mode == "periodic":
        return i % n
    if mode == "zero":
        return torch.where((i >= 0) & (i < n), i, torch.full_like(i, -1))
    r = i % (2 * n)
    return torch.where(r < n, r, 2 * n - 1 - r)


def _take(A, axis, idx):
    out = A.index_select(axis, idx.clamp(min=0))
    if bool((idx < 0).any()):
        shape = [1] * A.dim()
        shape[axis] = -1
        out = out * (idx >= 0).to(A.dtype).reshape(shape)
    return out


def _extended(V, n, mode):
    maps = []
    for a in range(3):
        i = torch.arange(-(n // 2), V.shape[a] + n // 2 - 1, device=V.device)
        maps.append(_ext(i, V.shape[a], mode))
    W = V
    for a in range(3):
        W = _take(W, a, maps[a])
    return W, maps


def _ratios(n, feature):
    """r_m / n^3 of every bin of the half spectrum (the half along the last axis, y), and its multiplicity."""
    f = torch.tensor([k if k < n // 2 else k - n for k in range(n)], dtype=F8, device="cuda")
    i, j, k = f[:, None, None] ** 2, f[None, :, None] ** 2, f[None, None, : n // 2 + 1] ** 2
    tot = i + j + k
    tot[0, 0, 0] = 1.0
    r = [((p if feature == "energy" else p.sqrt()) / (tot if feature == "energy" else tot.sqrt())).expand(n, n, n // 2 + 1).clone()
         for p in (j + k, i + k, i + j)]
    for a in r:
        a[0, 0, 0] = 0.0
    mult = torch.full((n // 2 + 1,), 2.0, dtype=F8, device="cuda")
    mult[0] = mult[-1] = 1.0
    return torch.stack([a / n ** 3 for a in r]), mult


def _cubes(Vx, n, taper, T, X, Y, stride):
    """Every cube, a batch of x rows at a time: (t0, x0 slice, cubes [x][y][n][n][n])."""
    per = max(1, int(6e7 // (len(range(0, Y, stride)) * n ** 3)))
    h = (0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(n, dtype=F8, device="cuda") / n)) if taper == "hann" else None
    xs = list(range(0, X, stride))
    for t in range(0, T, stride):
        for a in range(0, len(xs), per):
            sub = Vx[t : t + n, xs[a] : xs[min(a + per, len(xs)) - 1] + n]
            c = sub.unfold(1, n, stride).unfold(2, n, stride)        # [t][x][y][n_x][n_y]
            c = c.permute(1, 2, 0, 3, 4)
            yield t, xs[a : a + per], (c * h[:, None, None] * h[None, :, None] * h[None, None, :] if h is not None else c)


def _features(V, case):
    n, s = case["n"], case["stride"]
    T, X, Y = V.shape
    Vx, _ = _extended(V, n, case["boundary"])
    r, mult = _ratios(n, case["feature"])
    w = (r * mult).reshape(3, -1).T.contiguous()
    Tc, Xc, Yc = (-(-v // s) for v in (T, X, Y))
    E = torch.empty((3, Tc, Xc, Yc), dtype=F8, device="cuda")
    for t, xs, c in _cubes(Vx, n, case["taper"], T, X, Y, s):
        F = torch.fft.rfftn(c, dim=(2, 3, 4)).abs()
        if case["feature"] == "energy":
            F = F.square()
        E[:, t // s, xs[0] // s : xs[-1] // s + 1] = (F.reshape(len(xs), Yc, -1) @ w).permute(2, 0, 1)
    for a, (v, vc) in enumerate(((T, Tc), (X, Xc), (Y, Yc))):
        if s > 1:   # linear interpolation between lattice points, held past the last
            i = torch.arange(v, device="cuda")
            lo = i // s
            f = ((i % s).to(F8) / s) * (lo + 1 < vc)
            shape = [1, 1, 1, 1]
            shape[a + 1] = -1
            f = f.reshape(shape)
            E = E.index_select(a + 1, lo) * (1 - f) + E.index_select(a + 1, (lo + 1).clamp(max=vc - 1)) * f
    return E


def _window(case, alpha=(1.0, 1.0, 1.0)):
    out = []
    for d, v in enumerate(SECTION_DIRECTIONS if case["section"] else VOLUME_DIRECTIONS):
        for k in range(-R, R + 1):
            if k:
                o = tuple(k * c for c in v)
                g = math.exp(-sum(c * c for c in o) / (2 * SIGMA * SIGMA))
                out.append((o, g, d, float(np.float32(alpha[d])) * float(np.float32(g))))
    return out


def _neighbour(E, o, mode):
    for a in range(3):
        if o[a] or mode == "zero":
            i = torch.arange(E.shape[a + 1], device=E.device) + o[a]
            E = _take(E, a + 1, _ext(i, E.shape[a + 1], mode))
    return E


def _surround(E, case, alpha=(1.0, 1.0, 1.0)):
    win = _window(case, alpha)
    S3 = torch.zeros_like(E)
    for o, _, _, w in win:
        S3 += (E - w * _neighbour(E, o, case["boundary"])).abs()
    return S3 / len(win)


def _bounds(A):
    lo, hi = float(A.min()), float(A.max())
    return lo, (1.0 / (hi - lo) if hi - lo > 1e-30 * max(1.0, abs(hi)) else 0.0)


def _combined(S3, W, D=None):
    x = torch.stack([(S3[m] - lo) * inv for m, (lo, inv) in enumerate(_bounds(S3[m]) for m in range(3))])
    if D is not None:
        f = x.reshape(3, -1)
        W = torch.linalg.solve(f @ f.T + 1e-6 * torch.eye(3, dtype=F8, device="cuda"), f @ D.reshape(-1).to(F8))
    else:
        W = torch.tensor([float(np.float32(v)) for v in W], dtype=F8, device="cuda")
    C = (W[:, None, None, None] * x).sum(0)
    lo, inv = _bounds(C)
    return (C - lo) * inv, W, inv, x


def _adjoint(V, gE, case):
    n = case["n"]
    T, X, Y = V.shape
    Vx, maps = _extended(V, n, case["boundary"])
    r, _ = _ratios(n, case["feature"])
    r = r.reshape(3, -1)
    h = (0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(n, dtype=F8, device="cuda") / n)) if case["taper"] == "hann" else None
    out = torch.zeros_like(Vx)
    for t, xs, c in _cubes(Vx, n, case["taper"], T, X, Y, 1):
        F = torch.fft.rfftn(c, dim=(2, 3, 4))
        rho = (gE[:, t, xs[0] : xs[-1] + 1].permute(1, 2, 0) @ r).reshape(F.shape)
        if case["feature"] == "energy":
            G = 2.0 * rho * F
        else:
            m = F.abs()
            band = c.abs().sum((2, 3, 4), keepdim=True) * 2.0 ** -40    # a bin that is zero has no direction
            G = torch.where(m > band, rho / m.clamp(min=1e-300), torch.zeros_like(rho)) * F
        g = torch.fft.irfftn(G, s=(n, n, n), dim=(2, 3, 4)) * n ** 3
        if h is not None:
            g = g * h[:, None, None] * h[None, :, None] * h[None, None, :]
        B = len(xs)
        gy = torch.zeros((B, n, n, Y + n - 1), dtype=F8, device="cuda")
        for u in range(n):
            gy[..., u : u + Y] += g[..., u].permute(0, 2, 3, 1)
        for u in range(n):
            out[t : t + n, xs[0] + u : xs[-1] + 1 + u] += gy[:, :, u].permute(1, 0, 2)
    for a in range(3):
        idx = maps[a]
        keep = idx >= 0
        shape = list(out.shape)
        shape[a] = V.shape[a]
        out = torch.zeros(shape, dtype=F8, device="cuda").index_add_(a, idx[keep], out.index_select(a, keep.nonzero()[:, 0]))
    return out


def _surround_adjoint(E, gS3, case, alpha=(1.0, 1.0, 1.0)):
    win, mode = _window(case, alpha), case["boundary"]
    gE = torch.zeros_like(E)
    galpha = [0.0, 0.0, 0.0]
    for o, g, d, w in win:
        nb = _neighbour(E, o, mode)
        s = torch.sign(E - w * nb) * gS3
        gE += s
        galpha[d] -= float((s * nb).sum()) * g
        back = -w * s
        for a in range(3):
            n = E.shape[a + 1]
            idx = _ext(torch.arange(n, device="cuda") + o[a], n, mode)
            keep = idx >= 0
            back = torch.zeros_like(E).index_add_(a + 1, idx[keep], back.index_select(a + 1, keep.nonzero()[:, 0]))
        gE += back
    return gE / len(win), torch.tensor(galpha, dtype=F8) / len(win)


def _filter(S3, D, case):
    """The filters one voxel after the other, y outermost, then x, then t, in Python's own doubles."""
    T, X, Y = D.shape
    x = torch.stack([(S3[m].to(F8) - float(np.float32(lo))) * float(np.float32(1) / (np.float32(hi) - np.float32(lo)))
                     for m, (lo, hi) in enumerate((float(S3[m].min()), float(S3[m].max())) for m in range(3))])
    f = x.permute(3, 2, 1, 0).reshape(-1, 3).cpu().numpy()
    d = D.to(F8).permute(2, 1, 0).reshape(-1).cpu().numpy()
    sec = case["block"] or Y
    W, err = [], np.empty(d.size)
    for y0 in range(0, Y, sec):
        a, b = y0 * X * T, min(Y, y0 + sec) * X * T
        xs, ds, es = f[a:b].tolist(), d[a:b].tolist(), []
        if case["method"] == "rls":
            w, P = np.zeros(3), np.eye(3) / 1e-6
            for v, dv in zip(f[a:b], ds):
                e = dv - float(w @ v)
                es.append(e * e)
                Pv = P @ v
                k = Pv / (1.0 + float(v @ Pv))
                w = w + k * e
                P = P - np.outer(k, v @ P)
            w0, w1, w2 = w
        else:
            w0 = w1 = w2 = 1.0 / 3.0
            nlms = case["method"] == "nlms"
            for (p, q, r), dv in zip(xs, ds):
                e = dv - (w0 * p + w1 * q + w2 * r)
                es.append(e * e)
                g = 0.5 * e / (1e-8 + (p * p + q * q + r * r)) if nlms else 0.5 * e
                w0 += g * p
                w1 += g * q
                w2 += g * r
        err[a:b] = es
        W.append((w0, w1, w2))
    return {"W": np.array(W), "err2": err}


def exact(case, seed):
    N, kind = case["T"] * case["X"] * case["Y"], case["kind"]
    if kind in ("adapt", "dcs"):
        S3, D = _maps(case, seed)
        if kind == "adapt":
            return _filter(S3, D, case)
        gE, galpha = _surround_adjoint(S3.to(F8), _gradient(case, seed, 3).to(F8), case)
        return {"gE": gE, "galpha": galpha}
    cubes = N / case["stride"] ** 3
    if cubes * case["n"] ** 3 * (2 if kind == "adjoint" else 1) > WINDOW_COST:
        return None
    V, D = _volume(case, seed)
    V8 = V.to(F8)
    if kind == "adjoint":
        return {"gV": _adjoint(V8, _gradient(case, seed, 3).to(F8), case)}
    alpha = [float(np.float32(v)) for v in (1.0, 0.9, 1.1)] if kind == "fit" else (1.0, 1.0, 1.0)
    E = _features(V8, case)
    S3 = _surround(E, case, alpha)
    if kind == "forward":
        W = _weights(case) if case["weights"] == "given" else (1 / 3,) * 3
        S, W, _, _ = _combined(S3, W, D if case["weights"] == "template" else None)
        return {"S": S, "W": W, "E": E, "S3": S3}
    W = _weights(case)
    S, W, invC, x = _combined(S3, W)
    gS = (S - D.to(F8)) / N
    gW = torch.stack([(gS * x[m]).sum() * invC for m in range(3)])
    coef = torch.stack([W[m] * invC * _bounds(S3[m])[1] for m in range(3)])
    _, galpha = _surround_adjoint(E, coef[:, None, None, None] * gS, case, alpha)
    return {"S": S, "loss": 0.5 * (S - D.to(F8)).square().mean(), "gW": gW, "galpha": galpha}
