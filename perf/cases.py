"""The performance cases of the library: what its users have it do, over the sizes they do it at.

A case is one call sequence through the public binding:

  twoset_solve      points -> K x k modes by the paper's two-set construction (the splat route)
  nodal_solve       particles -> n x k modes by the nodal discretisation
  batch             many objects in one eigenmodes_batched call
  twoset_operators  points -> H_w and M of the two-set construction, applied to a block
  nodal_operators   particles -> H_w and M of the nodal discretisation, applied to a block
  apply             H_w and M of an assembled cloud applied to a block (a caller's own solver)
  matfree           the same without assembled matrices
  weights           skinning weight fields of the modes at the points to be skinned
  lbs               one frame of linear blend skinning at those points

Sizes are those of the benchmark's workloads, the tests and the batch configuration: nodal clouds
of 2,000 to 200,000 particles, two-set clouds of up to 1,000,000 points on up to 1,000 centres,
up to 64 modes; FP32 and FP64 contexts, and the FP32 build of an FP64 context.

The modes of a solve are handed on as a reduced simulation takes them: in FP32, each with its
free sign fixed.  FP64 builds are solved to a residual of 1e-7, a decade under the default as in
the tests, which makes the modes good to FP32; the FP32 build of the splat keeps the benchmark's
options.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_29318_gb300 import binding, synth

DEV = "cuda:0"

# what a pair of the two-set lists and of the nodal lists stands for: covering centres of a point
# (cut at 3 r_k) and nodes covering a particle (support 2.0 x spacing), and matrix entries of a
# nodal row
TWOSET_COVER = 98
NODAL_COVER = 33
NODAL_ROW = 160


def listed():
    return [
        # the headline: a splat scene's subspace, with the precision plan the benchmark gives it
        {"name": "splat1m_solve", "op": "twoset_solve", "cloud": "splat", "points": 1_000_000,
         "K": 1000, "k": 64, "build": "fp32", "tol": 1e-6, "cheb": 32, "fp32_tol": 3e-5},
        # the headline of the nodal discretisation: one particle object, default options
        {"name": "torus50k_solve", "op": "nodal_solve", "shape": "torus", "n": 50_000, "k": 32,
         "tol": 1e-7},
        # a small interactive object: the latency of a whole solve
        {"name": "object3k_solve", "op": "nodal_solve", "shape": "layers", "n": 3_001, "k": 10,
         "tol": 1e-7},
        # an asset library: objects of mixed size solved together
        {"name": "batch8_solve", "op": "batch", "count": 8, "nmin": 2_000, "nmax": 20_000,
         "kmin": 16, "kmax": 48, "tol": 1e-7},
        # a mesh object's inside grid, FP64 throughout, for a caller's own eigensolver
        {"name": "grid228k_operators", "op": "twoset_operators", "cloud": "torusgrid",
         "points": 228_000, "K": 1000, "m": 8, "prec": "fp64"},
        # the largest nodal cloud of the batch configuration, in the default precision
        {"name": "cloud200k_operators", "op": "nodal_operators", "shape": "ellipsoids",
         "n": 200_000, "m": 8, "prec": "fp32"},
        # the smallest call: the operators of a small object on a few vectors
        {"name": "apply2k_fp32", "op": "apply", "shape": "cube", "n": 2_000, "m": 10,
         "prec": "fp32"},
        # one block product of a caller's own block solver in FP64
        {"name": "apply50k_fp64", "op": "apply", "shape": "torus", "n": 50_000, "m": 40,
         "prec": "fp64"},
        # the same without assembled matrices (per-particle material)
        {"name": "matfree30k_fp32", "op": "matfree", "shape": "layers", "n": 30_011, "m": 32,
         "prec": "fp32"},
        # weight fields of a nodal object's modes at its particles, in FP64
        {"name": "weights50k_fp64", "op": "weights", "cloud": "torus", "n": 50_000,
         "nq": 50_000, "m": 32, "prec": "fp64"},
        # weight fields of a splat scene's modes at every Gaussian
        {"name": "weights1m_fp32", "op": "weights", "cloud": "splat", "points": 1_000_000,
         "K": 1000, "nq": 1_000_000, "m": 64, "prec": "fp32"},
        # a frame of the animation: every Gaussian of the scene skinned
        {"name": "lbs1m_fp32", "op": "lbs", "nq": 1_000_000, "m": 64, "prec": "fp32"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["twoset_solve", "nodal_solve", "batch", "twoset_operators",
                     "nodal_operators", "apply", "matfree", "weights", "lbs"])
    prec = rng.choice(["fp32", "fp64"])
    shape = rng.choice(["cube", "torus", "ellipsoids", "layers"])
    if op == "twoset_solve":
        build = rng.choice(["fp32", "fp64"])
        c = {"op": op, "cloud": "splat",
             "points": _logint(rng, 20_000, 1_000_000 if build == "fp32" else 200_000),
             "K": _logint(rng, 150, 1000), "k": rng.randint(8, 64), "build": build,
             "tol": 1e-6 if build == "fp32" else 1e-7}
        if build == "fp32":
            c.update(cheb=32, fp32_tol=3e-5)
        return c
    if op == "nodal_solve":
        return {"op": op, "shape": shape, "n": _logint(rng, 2_000, 50_000),
                "k": rng.randint(8, 40), "tol": 1e-7}
    if op == "batch":
        return {"op": op, "count": rng.randint(3, 8), "nmin": 2_000,
                "nmax": _logint(rng, 4_000, 20_000), "kmin": 16, "kmax": 48, "tol": 1e-7}
    if op == "twoset_operators":
        return {"op": op, "cloud": rng.choice(["splat", "torusgrid"]),
                "points": _logint(rng, 8_000, 228_000), "K": _logint(rng, 100, 1000),
                "m": rng.randint(1, 16), "prec": prec}
    if op == "nodal_operators":
        return {"op": op, "shape": shape, "n": _logint(rng, 2_000, 200_000),
                "m": rng.randint(1, 16), "prec": prec}
    if op in ("apply", "matfree"):
        return {"op": op, "shape": shape, "n": _logint(rng, 2_000, 50_000),
                "m": rng.randint(1, 64), "prec": prec}
    if op == "weights":
        if rng.random() < 0.5:
            return {"op": op, "cloud": shape, "n": _logint(rng, 2_000, 50_000),
                    "nq": _logint(rng, 1_000, 200_000), "m": rng.randint(4, 64), "prec": prec}
        return {"op": op, "cloud": "splat", "points": _logint(rng, 20_000, 200_000),
                "K": _logint(rng, 150, 1000), "nq": _logint(rng, 1_000, 200_000),
                "m": rng.randint(4, 64), "prec": prec}
    return {"op": op, "nq": _logint(rng, 1_000, 1_000_000), "m": rng.randint(4, 64),
            "prec": prec}


# ------------------------------------------------------------------ inputs
def _nodal(shape, n, seed):
    """A nodal cloud of the shape as device arrays; supports floored at 1.5 times the distance
    of the 8 nearest, as the batch configuration does, so that any seed covers every particle."""
    make = {"cube": synth.unit_cube, "torus": synth.torus, "layers": synth.layered_sphere,
            "ellipsoids": synth.ellipsoid_union}[shape]
    c = make(n, seed=1000 + seed)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    d = {"X": torch.from_numpy(c.X).to(DEV), "v": torch.from_numpy(c.v).to(DEV),
         "a": torch.from_numpy(a).to(DEV), "E": None, "nu": None, "E0": 1.0, "nu0": float(c.nu)}
    if np.ndim(c.E):
        d["E"] = torch.from_numpy(c.E).to(DEV)
    else:
        d["E0"] = float(c.E)
    return d


def _splat(n, seed, n_comp=64):
    """A splat-like cloud after synth.gaussian_mixture, drawn on the GPU: the mixture's own
    density at a point gives its volume, 1 / (n p(x))."""
    rng = np.random.default_rng(seed)
    scales = np.exp(rng.uniform(np.log(0.02), np.log(0.3), size=(n_comp, 3)))
    rots = np.stack([np.linalg.qr(rng.normal(size=(3, 3)))[0] for _ in range(n_comp)])
    centres = np.zeros((n_comp, 3))
    for c in range(1, n_comp):
        two = np.sort(scales[c - 1])[-2:].sum() + np.sort(scales[c])[-2:].sum()
        step = rng.normal(size=3)
        centres[c] = centres[c - 1] + 0.35 * two * step / np.linalg.norm(step)
    modulus = np.exp(rng.uniform(np.log(1e4), np.log(1e7), size=n_comp))
    g = torch.Generator(device=DEV).manual_seed(seed)
    s, R, o, Ec = (torch.from_numpy(x).float().to(DEV) for x in (scales, rots, centres, modulus))
    comp = torch.randint(n_comp, (n,), generator=g, device=DEV)
    Z = torch.randn((n, 3), generator=g, device=DEV)
    Z = torch.where(Z.abs() > 3.0, torch.remainder(Z, 3.0), Z)
    X = o[comp] + torch.einsum("ni,nji->nj", Z * s[comp], R[comp])
    lognorm = -s.log().sum(1) - 1.5 * math.log(2 * math.pi) - math.log(n_comp)
    logp = torch.empty(n, device=DEV)
    for b in range(0, n, 1 << 16):
        e = torch.einsum("bci,cij->bcj", X[b:b + (1 << 16), None] - o, R) / s
        logp[b:b + (1 << 16)] = torch.logsumexp(lognorm - 0.5 * e.square().sum(2), 1)
    return {"X": X.contiguous(), "v": torch.exp(-logp) / n, "E": Ec[comp].contiguous(),
            "nu": None, "E0": 1.0, "nu0": 0.45}


def _torus_grid(points, seed):
    """The solid torus's inside grid of about that many points, in a pose of the seed's."""
    R, r = 0.5, 0.2
    h = (2 * math.pi ** 2 * R * r * r / points) ** (1 / 3)
    rng = np.random.default_rng(seed)
    off = h * rng.random(3)

    def inside(P):
        rho = np.sqrt(P[:, 0] ** 2 + P[:, 1] ** 2)
        return (rho - R) ** 2 + P[:, 2] ** 2 < r * r
    X, v = synth.inside_grid([-R - r - off[0], -R - r - off[1], -r - off[2]],
                             [R + r + h, R + r + h, r + h], h, inside)
    return {"X": torch.from_numpy(X).to(DEV), "v": torch.from_numpy(v).to(DEV), "E": None,
            "nu": None, "E0": 1e6, "nu0": 0.4}


def _cloud(case, seed):
    name = case.get("cloud") or case["shape"]
    if name == "splat":
        return _splat(case["points"], seed)
    if name == "torusgrid":
        return _torus_grid(case["points"], seed)
    return _nodal(name, case["n"], seed)


def _dtype(prec):
    return torch.float64 if prec == "fp64" else torch.float32


def _randn(shape, seed, dtype):
    g = torch.Generator(device=DEV).manual_seed(7919 * seed + 13)
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32).to(dtype)


def _queries(case, cloud, seed):
    """Points to be skinned: the cloud's own points, and, where more are asked for, points a
    little off them."""
    X, nq = cloud["X"], case["nq"]
    at = torch.arange(nq, device=DEV) % X.shape[0]
    Q = X[at].clone()
    if nq > X.shape[0]:
        ext = (X.max(0).values - X.min(0).values).max()
        Q[X.shape[0]:] += 1e-3 * ext * _randn((nq - X.shape[0], 3), seed + 1, torch.float32)
    return Q.contiguous()


def _build(ctx, s):
    if "K" in s["case"]:
        ctx.rkpm_build_twoset(s["X"], s["v"], s["case"]["K"], 3.0, 0)
    else:
        ctx.rkpm_build(s["X"], s["v"], s["a"])


def prepare(case, seed):
    op = case["op"]
    s = {"case": dict(case)}
    if op == "lbs":
        t = _dtype(case["prec"])
        s["ctx"] = binding.Context(0, case["prec"])
        s["Q"] = _randn((case["nq"], 3), seed, torch.float32)
        W = _randn((case["nq"], case["m"]), seed + 1, torch.float32)
        s["W"] = (W / case["m"]).to(t).contiguous()
        s["Z"] = (0.1 * _randn((case["m"], 3, 4), seed + 2, torch.float32)).to(t).contiguous()
        return s
    if op == "batch":
        s["objects"], s["probes"] = [], []
        for j in range(case["count"]):
            t = j / max(1, case["count"] - 1)
            n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** t))
            d = _nodal(("cube", "torus", "ellipsoids")[j % 3], n, 100 * seed + j)
            d["k"] = case["kmax"] - round(t * (case["kmax"] - case["kmin"]))
            s["objects"].append(d)
            s["probes"].append(_randn((n,), 100 * seed + j, torch.float64))
        s["opts"] = binding.default_opts(tol=case["tol"])
        return s
    s.update(_cloud(case, seed))
    if op in ("twoset_solve", "nodal_solve"):
        s["ctx"] = binding.Context(0, "fp64")
        if case.get("build") == "fp32":
            s["ctx"].set_build_precision("fp32")
        s["opts"] = binding.default_opts(**{name: case[key] for name, key in
                                            (("tol", "tol"), ("cheb_degree", "cheb"),
                                             ("fp32_tol", "fp32_tol"))
                                            if key in case})
        s["probe"] = _randn((case.get("K") or case["n"],), seed, torch.float64)
        return s
    s["ctx"] = binding.Context(0, case["prec"])
    n = case.get("K") or case["n"]
    s["B"] = _randn((n, case["m"]), seed, _dtype(case["prec"]))
    if op in ("twoset_operators", "nodal_operators"):
        return s
    _build(s["ctx"], s)
    if op == "apply":
        s["ctx"].assemble_hessian(s["E"], s["nu"], s["E0"], s["nu0"])
    if op == "weights":
        s["Q"] = _queries(case, s, seed)
    return s


# ------------------------------------------------------------------ the calls
def _signed(modes, probe):
    """The modes (n, k) in FP32 as a simulation takes them, each with the sign that makes its
    product with the probe positive."""
    sign = torch.where(probe @ modes < 0, -1.0, 1.0)
    return (modes * sign).float()


# a solve whose residual levels off above the tolerance still hands on its best block
_USABLE = (0, 5)


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "lbs":
        return s["ctx"].lbs(s["Q"], s["W"], s["Z"])
    if op == "batch":
        _, res = binding.eigenmodes_batched(s["objects"], "fp64", s["opts"])
        if any(r[3] not in _USABLE for r in res):
            raise RuntimeError([r[3:] for r in res])
        return [{"eigvals": r[0], "modes": _signed(r[1], p)} for r, p in zip(res, s["probes"])]
    ctx = s["ctx"]
    if op == "weights":
        return ctx.skinning_weights(s["Q"], s["B"])
    if op == "apply":
        return ctx.apply_operators(s["B"])
    if op == "matfree":
        return ctx.apply_operators_matfree(s["B"], s["E"], s["nu"], s["E0"], s["nu0"])
    _build(ctx, s)
    ctx.assemble_hessian(s["E"], s["nu"], s["E0"], s["nu0"])
    if op in ("twoset_operators", "nodal_operators"):
        return ctx.apply_operators(s["B"])
    ev, modes, _, st = ctx.eigenmodes(case["k"], s["opts"], check=False)
    if st not in _USABLE:
        raise RuntimeError(binding.STATUS[st])
    # an FP32 build carries its eigenvalues to FP32
    return {"eigvals": ev.astype(np.float32) if case.get("build") == "fp32" else ev,
            "modes": _signed(modes, s["probe"])}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    op = case["op"]
    if op == "lbs":
        e = 8 if case["prec"] == "fp64" else 4
        nq, m = case["nq"], case["m"]
        return {"bytes": nq * (12 + e * (m + 3)) + 12 * e * m, "flops": 24.0 * nq * m}
    if op == "batch":
        n = math.sqrt(case["nmin"] * case["nmax"]) * case["count"]
        k = 0.5 * (case["kmin"] + case["kmax"])
        return {"bytes": n * (20 + 8 * k + 12 * NODAL_ROW), "flops": n * NODAL_COVER ** 2 * 8}
    twoset = "K" in case
    n = case["K"] if twoset else case["n"]
    pts = case["points"] if twoset else n
    cover = min(TWOSET_COVER, n) if twoset else NODAL_COVER
    e = 4 if case.get("prec") == "fp32" else 8
    entries = min(n * n, 376 * n) if twoset else n * NODAL_ROW
    if op == "weights":
        nq, m = case["nq"], case["m"]
        return {"bytes": nq * (12 + e * m) + n * (e * m + 16),
                "flops": nq * cover * (150.0 + 2 * m)}
    if op == "apply":
        return {"bytes": entries * (4 + 2 * e) + 3 * n * case["m"] * e,
                "flops": 4.0 * entries * case["m"]}
    if op == "matfree":
        return {"bytes": pts * cover * (4 + 4 * e) + 3 * n * case["m"] * e,
                "flops": 16.0 * pts * cover * case["m"]}
    # a build: the points in, the shape functions and pair products, the matrices out once; a
    # solve: the modes out besides
    out = (2 * n * case["m"] * e + n * case["m"] * e if op.endswith("operators")
           else 4 * n * case["k"])
    return {"bytes": pts * 20 + entries * (4 + 2 * e) + out,
            "flops": pts * (cover * 150.0 + cover * cover * 8.0 / 2)}


# ------------------------------------------------------------------ 64-bit values
def _kernel(case, d2, P_r):
    """Raw kernel and gs (its gradient is gs (p - x)) of squared distances in FP64: the cubic
    B-spline of radius P_r, or the Gaussian of radius P_r."""
    if "K" in case:
        w = torch.exp(-d2 / P_r ** 2)
        return w, 2 * w / P_r ** 2
    q = d2.sqrt() / P_r
    t = (1 - q).clamp_min(0)
    near = q <= 0.5
    w = torch.where(near, 2 / 3 - 4 * q * q + 4 * q ** 3, 4 / 3 * t ** 3)
    dwq = torch.where(near, -8 + 12 * q, -4 * t * t / q.clamp_min(0.5))
    return w, -dwq / P_r ** 2


def _tables(case, Q, P, r):
    """Corrected shape functions of the nodes P (radii r; Gaussians are cut at 3 r) at the points
    Q in FP64: (point, node, phi, dphi) of every covering pair.  Nodal clouds come sorted along
    x, so that a block of points needs a window of nodes only."""
    out = []
    n = P.shape[0]
    cut = 9.0 if "K" in case else 1.0
    if "K" in case:
        blocks = [(a, min(a + 8192, Q.shape[0]), 0, n) for a in range(0, Q.shape[0], 8192)]
    else:
        blocks = []
        rmax = float(r.max())
        size = max(64, min(2048, Q.shape[0] // 64))
        px = P[:, 0].contiguous()
        for a in range(0, Q.shape[0], size):
            b = min(a + size, Q.shape[0])
            lo = int(torch.searchsorted(px, Q[a, 0] - rmax))
            hi = int(torch.searchsorted(px, Q[b - 1, 0] + rmax))
            blocks.append((a, b, lo, hi))
    for a, b, lo, hi in blocks:
        d = P[None, lo:hi] - Q[a:b, None]                        # (b, n, 3)
        e = d.square()
        d2 = e[..., 0] + e[..., 1] + e[..., 2]
        rb = r[None, lo:hi]
        at = torch.nonzero(d2 < cut * (rb * rb), as_tuple=True)
        w, gs = _kernel(case, d2[at], r[lo + at[1]])
        d = d[at]
        out.append((at[0] + a, at[1] + lo, w, gs, d))
    i = torch.cat([o[0] for o in out])
    k = torch.cat([o[1] for o in out])
    w, gs, d = (torch.cat([o[j] for o in out]) for j in (2, 3, 4))
    del out
    nq = Q.shape[0]
    scale = float(r.mean())
    p = torch.cat([torch.ones_like(d[:, :1]), d / scale], 1)
    M = torch.zeros((nq, 4, 4), dtype=torch.float64, device=DEV)
    dM = torch.zeros((3, nq, 4, 4), dtype=torch.float64, device=DEV)
    for x in range(4):
        for y in range(4):
            pp = p[:, x] * p[:, y]
            M[:, x, y].index_add_(0, i, w * pp)
            for t in range(3):
                dM[t, :, x, y].index_add_(0, i, gs * d[:, t] * pp)
    e0 = torch.zeros((nq, 4), dtype=torch.float64, device=DEV)
    e0[:, 0] = 1
    C = torch.linalg.solve(M, e0)
    phi = w * (p * C[i]).sum(1)
    dphi = []
    for t in range(3):
        rhs = -(dM[t] @ C[:, :, None])[:, :, 0]
        rhs[:, 1 + t] += 1 / scale
        dC = torch.linalg.solve(M, rhs)
        dphi.append(gs * d[:, t] * (p * C[i]).sum(1) + w * (p * dC[i]).sum(1))
    return i, k, phi, dphi


def _centres(X, K):
    """Farthest-point centres from point 0 and their radii (second-nearest centre)."""
    X = X.double()
    near = torch.full((X.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    last = torch.zeros((), dtype=torch.int64, device=DEV)
    cen = [last]
    for _ in range(K - 1):
        e = (X - X[last]).square()
        near = torch.minimum(near, e[:, 0] + e[:, 1] + e[:, 2])
        last = near.argmax()
        cen.append(last)
    P = X[torch.stack(cen)]
    e = (P[:, None] - P[None]).square()
    d2 = e[..., 0] + e[..., 1] + e[..., 2]
    return P, d2.topk(3, dim=1, largest=False).values[:, 2].sqrt()


def _nodes(case, d):
    """Nodes, radii and their order of a cloud (nodal ones sorted along x)."""
    if "K" in case:
        P, r = _centres(d["X"], case["K"])
        return P, r, torch.arange(case["K"], device=DEV)
    order = d["X"][:, 0].argsort()
    return d["X"][order].double(), d["a"][order].double(), order


def _material(d):
    E = d["E"].double() if d["E"] is not None else d["E0"]
    nu = d["nu"].double() if d["nu"] is not None else d["nu0"]
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    return d["v"].double() * (lam + 4 * mu)


def _operators(case, d, B):
    """H_w B and M B in FP64, point block by point block."""
    P, r, order = _nodes(case, d)
    Q, v, wh = d["X"].double(), d["v"].double(), _material(d)
    if "K" not in case:
        Q, v, wh = Q[order], v[order], wh[order]
    Bo = B.double()[order]
    YH, YM = torch.zeros_like(Bo), torch.zeros_like(Bo)
    step = 100_000 if "K" in case else Q.shape[0]
    for a in range(0, Q.shape[0], step):
        i, k, phi, dphi = _tables(case, Q[a:a + step], P, r)
        for tab, wt, Y in ((phi, v, YM), *((g, wh, YH) for g in dphi)):
            G = torch.sparse_coo_tensor(torch.stack([i, k]), tab,
                                        (min(step, Q.shape[0] - a), P.shape[0]))
            Y += torch.sparse.mm(G.t(), wt[a:a + step, None] * torch.sparse.mm(G, Bo))
    back = order.argsort()
    return YH[back], YM[back]


def _pencil_modes(case, d, k, probe):
    """The k lowest eigenpairs (constant mode first) of the dense pencil."""
    n = probe.numel()
    H, M = _operators(case, d, torch.eye(n, dtype=torch.float64, device=DEV))
    L = torch.linalg.cholesky(0.5 * (M + M.t()))
    A = torch.linalg.solve_triangular(L, 0.5 * (H + H.t()), upper=False)
    A = torch.linalg.solve_triangular(L, A.t().contiguous(), upper=False)
    ev, U = torch.linalg.eigh(0.5 * (A + A.t()))
    C = torch.linalg.solve_triangular(L.t(), U[:, :k], upper=True)
    ev = ev[:k].clone()
    ev[0] = 0
    C *= torch.where(probe @ C < 0, -1.0, 1.0)
    return ev.cpu().numpy(), C


def exact(case, seed):
    op = case["op"]
    # over about 20 seconds: the eigenvectors of large pencils
    if op == "batch":
        s = prepare(case, seed)
        out = []
        for d, p in zip(s["objects"], s["probes"]):
            ev, C = _pencil_modes(d, d, d["k"], p) if p.numel() <= 4_000 else (None, None)
            out.append({"eigvals": ev, "modes": C})
        return out
    if op == "nodal_solve" and case["n"] > 4_000:
        return None
    if op == "lbs":
        s = prepare(case, seed)
        Q, W, Z = s["Q"].double(), s["W"].double(), s["Z"].double()
        h = torch.cat([Q, torch.ones_like(Q[:, :1])], 1)
        T = (W @ Z.reshape(case["m"], 12)).reshape(-1, 3, 4)
        return Q + (T @ h[:, :, None])[:, :, 0]
    d = _cloud(case, seed)
    if op.endswith("solve"):
        probe = _randn((case.get("K") or case["n"],), seed, torch.float64)
        ev, C = _pencil_modes(case, d, case["k"], probe)
        return {"eigvals": ev, "modes": C}
    B = _randn((case.get("K") or case["n"], case["m"]), seed, _dtype(case["prec"]))
    if op == "weights":
        P, r, order = _nodes(case, d)
        Q = _queries(case, d, seed).double()
        Bo = B.double()[order]
        qorder = Q[:, 0].argsort()
        W = torch.zeros((Q.shape[0], case["m"]), dtype=torch.float64, device=DEV)
        step = 100_000
        for a in range(0, Q.shape[0], step):
            at = qorder[a:a + step]
            i, k, phi, _ = _tables(case, Q[at], P, r)
            G = torch.sparse_coo_tensor(torch.stack([i, k]), phi, (at.numel(), P.shape[0]))
            W[at] = torch.sparse.mm(G, Bo)
        return W
    return _operators(case, d, B)
