"""What this framework is used for, as cases that can be timed: Monte Carlo solves of variable-coefficient
elliptic problems through the public entry points of the Python binding (solve, solve_host, solve_grad,
solve_nf, solve_batch, SliceView.frame, autograd.CoefficientSolve).

A case names a problem of the workloads module, a number of points and of walks per point, and whether the
program compiled its kernels for the problem (Problem.specialize, which a program with one problem and many
solves does once) or runs the generic ones (a one-off solve).  FP32 walks throughout: the FP64 walks exist to
replay the oracle's walks in tests.

Walk steps per walk (STEPS) and operations per step (FLOPS) are properties of the problems and of the
method's arithmetic (one Philox block, one Green's-function sample, the coefficients), not of the kernels.
"""
import functools
import math

import numpy as np
import torch

import paper_2201_13240_gb300 as wos
import workloads as W
from paper_2201_13240_gb300.autograd import CoefficientSolve

# problem -> (mean steps of a walk, floating-point operations of a step with its coefficients)
STEPS = {"square2d": 10.5, "cube3d": 23.5, "literal": 25.2, "hifreq": 54.0, "noise_cube": 28.5,
         "noise_annulus": 12.7, "inverse": 24.3, "mesh": 95.0, "mesh_manufactured": 42.0, "csg": 8.0, "batch": 26.0}
FLOPS = {"square2d": 220.0, "cube3d": 330.0, "literal": 400.0, "hifreq": 220.0, "noise_cube": 900.0,
         "noise_annulus": 500.0, "inverse": 900.0, "mesh": 3000.0, "mesh_manufactured": 2500.0, "csg": 400.0,
         "batch": 500.0}
EPS = {"square2d": 1e-3, "hifreq": 1e-3, "noise_annulus": 1e-3, "batch": 1e-3}
LATTICE = {"square2d": 256, "hifreq": 256, "noise_annulus": 256, "mesh": 48, "mesh_manufactured": 48, "inverse": 48}
DIM2 = ("square2d", "hifreq", "noise_annulus", "batch")


def listed():
    return [
        # the first thing a user runs: config 1 (unit square, 32^2 points x 256 walks), generic kernel; a call of
        # a few hundred microseconds, where the launch and the longest walk count
        {"name": "square2d_small", "kind": "solve", "problem": "square2d", "points": 1024, "walks": 256, "spec": False},
        # one frame of the interactive view: one walk for each of 512^2 slice points of the CSG scene, and the image
        {"name": "slice_frame", "kind": "slice", "problem": "csg", "points": 512, "walks": 1, "spec": True,
         "width": 1280, "height": 720},
        # host buffers in and out, an odd number of scattered points and of walks
        {"name": "host_odd", "kind": "host", "problem": "cube3d", "points": 5003, "walks": 333, "spec": True},
        # config 2, the benchmark: 64^3 points x 1024 walks of the 3D drift problem, kernel compiled for it
        {"name": "cube3d_full", "kind": "solve", "problem": "cube3d", "points": 262144, "walks": 1024, "spec": True},
        # config 2 with its literal, non-conservative drift (the extra-drift walk)
        {"name": "literal_drift", "kind": "solve", "problem": "literal", "points": 46656, "walks": 300, "spec": True},
        # value and gradient at scattered points (the gradient walk)
        {"name": "gradient", "kind": "grad", "problem": "cube3d", "points": 32768, "walks": 512, "spec": True},
        # high-frequency diffusion with the weight window (roulette and splitting), generic kernel
        {"name": "weight_window", "kind": "window", "problem": "hifreq", "points": 4096, "walks": 256, "spec": False},
        # config 3: triangle mesh (327,680 triangles), certified-radius distance queries, 128^3 coefficient grids
        {"name": "mesh_tol", "kind": "solve", "problem": "mesh", "points": 8192, "walks": 100, "spec": True,
         "level": 7, "tol": 0.1},
        # the same walk with exact distance queries (the default) on a coarser mesh, generic kernel
        {"name": "mesh_exact", "kind": "solve", "problem": "mesh", "points": 3000, "walks": 64, "spec": False,
         "level": 5, "tol": 0.0},
        # config 4: many small 2D problems with their own 64^2 grids, uneven points and walks, one launch
        {"name": "batch", "kind": "batch", "problem": "batch", "problems": 192, "points": 4096, "walks": 1024,
         "spec": True},
        # config 5: one training step of the inverse problem, the estimates at 4096 sensors and the gradients of
        # a least-squares loss by both coefficient grids
        {"name": "inverse_step", "kind": "inverse", "problem": "inverse", "points": 4096, "walks": 512, "spec": True},
        # next-flight walks with the 8-term series kernels
        {"name": "next_flight", "kind": "nf", "problem": "cube3d", "points": 32768, "walks": 96, "spec": False,
         "terms": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, its problem, and sizes over the whole range (points from a handful to 64^3, walks
    per point from one to thousands), with no more walk steps than the largest listed case of the kind's cost."""
    kind = rng.choice(["solve", "solve", "solve", "host", "grad", "window", "mesh", "slice", "batch", "inverse", "nf"])
    spec = rng.random() < 0.6

    def sizes(most_points, most_walks, budget):
        p = _log(rng, 16, most_points)
        w = _log(rng, 8, most_walks)
        return p, max(1, min(w, budget // p))

    if kind in ("solve", "host"):
        prob = rng.choice(["square2d", "cube3d", "cube3d", "literal", "noise_cube", "noise_annulus"])
        p, w = sizes(262144, 8192, 40_000_000 if spec and prob in ("square2d", "cube3d", "literal") else 8_000_000)
        if kind == "host":
            p = min(p, 65536)
        return {"kind": kind, "problem": prob, "points": p, "walks": w, "spec": spec}
    if kind == "grad":
        p, w = sizes(65536, 2048, 16_000_000)
        return {"kind": kind, "problem": rng.choice(["cube3d", "square2d"]), "points": p, "walks": w, "spec": spec}
    if kind == "window":
        p, w = sizes(16384, 2048, 1_500_000)
        return {"kind": kind, "problem": "hifreq", "points": p, "walks": w, "spec": spec}
    if kind == "mesh":
        tol = rng.choice([0.0, 0.1, 0.1, 0.25])
        p, w = sizes(16384, 512, 150_000 if tol == 0.0 else 800_000)
        return {"kind": "solve", "problem": rng.choice(["mesh", "mesh_manufactured"]), "points": p, "walks": w,
                "spec": spec, "level": rng.randint(3, 6), "tol": tol}
    if kind == "slice":
        return {"kind": kind, "problem": "csg", "points": rng.randint(48, 512), "walks": rng.randint(1, 4), "spec": spec,
                "width": rng.choice([640, 961, 1280]), "height": rng.choice([360, 541, 720])}
    if kind == "batch":
        return {"kind": kind, "problem": "batch", "problems": _log(rng, 2, 160), "points": _log(rng, 64, 4096),
                "walks": _log(rng, 128, 1024), "spec": spec}
    if kind == "inverse":
        p, w = sizes(4096, 2048, 2_000_000)
        return {"kind": kind, "problem": "inverse", "points": p, "walks": w, "spec": spec}
    p, w = sizes(32768, 512, 3_000_000)
    return {"kind": "nf", "problem": rng.choice(["cube3d", "square2d"]), "points": p, "walks": w, "spec": False,
            "terms": rng.choice([0, 4, 8, 8, 16])}


# ---- what a program has in hand before the call ----
@functools.lru_cache(maxsize=None)
def _ctx():
    return wos.Context(0)


@functools.lru_cache(maxsize=4)
def _mesh(kind, level):
    # the mesh and its coefficient grids are a program's data, made once; the handle is made by prepare
    return W.mesh_noise_problem(level=level) if kind == "mesh" else W.mesh_manufactured_problem(level=level)


@functools.lru_cache(maxsize=4)
def _batch(problems, points, walks):
    return W.batch_problems(problems, seed=7, max_points=points, max_walks=walks)


def _describe(case):
    p = case["problem"]
    if p in ("mesh", "mesh_manufactured"):
        d = dict(_mesh(p, case["level"]))
        d["domain"] = dict(d["domain"], tol=case["tol"])
        return d
    return {"square2d": W.square2d_problem, "cube3d": W.cube3d_problem, "literal": W.cube3d_literal_problem,
            "hifreq": W.hifreq_alpha_problem, "noise_cube": W.noise_cube_problem,
            "noise_annulus": W.noise_annulus_problem, "csg": W.csg_variable_problem}[p]()


def _points(case, seed):
    """SoA float32 [dim][points]: cell centres where the count is a whole grid (as the benchmark's), else
    scattered points inside the domain."""
    p, n = case["problem"], case["points"]
    dim = 2 if p in DIM2 else 3
    if p in ("mesh", "mesh_manufactured"):
        return W.mesh_interior_points(n, seed)
    if p == "noise_annulus":
        rng = np.random.default_rng(seed)
        r, t = np.sqrt(rng.uniform(0.36 ** 2, 1.09 ** 2, n)), rng.uniform(0, 2 * np.pi, n)
        return np.stack([r * np.cos(t), r * np.sin(t)]).astype(np.float32)
    side = round(n ** (1.0 / dim))
    if side ** dim == n and p != "inverse":
        return W.cell_centres(dim, side)
    return W.uniform_in_box(dim, n, 0.02, 0.98, seed)


def prepare(case, seed):
    ctx, kind = _ctx(), case["kind"]
    st = {"kind": kind, "ctx": ctx, "seed": int(seed), "walks": case["walks"], "eps": EPS.get(case["problem"], 1e-4)}
    if kind == "batch":
        probs, pts, offs, walks = _batch(case["problems"], case["points"], case["walks"])
        hp = [ctx.problem(q) for q in probs]
        st["batch"] = ctx.batch(hp, offs, [ctx.sigma_bar(h, 64)[0] for h in hp])
        if case["spec"]:
            st["batch"].specialize(("fp32",))
        st["pts"], st["walks"] = torch.from_numpy(pts).cuda(), torch.from_numpy(walks).cuda()
        return st
    if kind == "inverse":
        st["sigma"] = torch.from_numpy(W.inverse_sigma_grid()).cuda()
        st["alpha"] = torch.from_numpy(W.inverse_alpha_grid()).cuda()
        desc = W.inverse_problem(st["sigma"].cpu().numpy(), st["alpha"].cpu().numpy())
        desc["sigma"], desc["alpha"] = dict(desc["sigma"], data=st["sigma"]), dict(desc["alpha"], data=st["alpha"])
        rng = np.random.default_rng(seed)
        st["target"] = torch.from_numpy(rng.uniform(1.0, 2.0, case["points"])).cuda()
        for k in ("sigma", "alpha"):
            st[k].requires_grad_(True)
    else:
        desc = _describe(case)
    st["prob"] = ctx.problem(desc)
    if case["spec"]:
        variant = {"grad": "grad", "window": "window"}.get(kind, "plain")
        st["prob"].specialize(("fp32",), ("plain", "adjoint") if kind == "inverse" else (variant,))
    st["sb"] = ctx.sigma_bar(st["prob"], LATTICE.get(case["problem"], 64))[0]
    if kind == "slice":
        n = case["points"]
        v = wos.view([-1.3, -1.3, 0.05], [2.6, 0, 0], [0, 2.6, 0], n, n, case["width"], case["height"], (-3.0, 3.0),
                     eye=(2.5, 2.0, 3.5), look=(0, 0, 0))
        st["view"] = wos.SliceView(ctx, st["prob"], v, st["eps"], st["sb"], seed=seed)
        return st
    pts = torch.from_numpy(_points(case, seed))
    st["pts"] = pts.pin_memory() if kind == "host" else pts.cuda()
    st["terms"] = case.get("terms", 0)
    return st


def run(st):
    """One pass.  Solves return what a program reads of them: mean, variance and standard error of each point's
    estimate, and its number of walks."""
    ctx, kind = st["ctx"], st["kind"]
    if kind == "slice":
        img = st["view"].frame(st["walks"])
        return [img] + list(st["view"].accum)
    if kind == "batch":
        acc, _ = ctx.solve_batch(st["batch"], st["pts"], st["walks"], st["eps"], seed=st["seed"])
        return list(ctx.finalize(acc)) + [acc[2]]
    a = (st["prob"], st["pts"], st["walks"], st["eps"], st["sb"])
    if kind == "host":
        return list(ctx.solve_host(*a, seed=st["seed"])[:3])
    if kind == "inverse":
        mean = CoefficientSolve.apply(st["sigma"], st["alpha"], ctx, *a, st["seed"])
        loss = (mean - st["target"]).square().mean()
        return [mean.detach()] + list(torch.autograd.grad(loss, (st["sigma"], st["alpha"])))
    if kind == "grad":
        acc, gacc, _ = ctx.solve_grad(*a, seed=st["seed"])
        return list(ctx.finalize(acc)) + list(ctx.finalize_grad(gacc, acc[2])) + [acc[2]]
    if kind == "nf":
        acc, _ = ctx.solve_nf(*a, seed=st["seed"], series_terms=st["terms"])
    else:
        acc, _ = ctx.solve(*a, seed=st["seed"], window=(0.5, 1.5) if kind == "window" else None)
    return list(ctx.finalize(acc)) + [acc[2]]


def work(case):
    kind, p = case["kind"], case["problem"]
    if kind == "batch":  # means of the log-uniform counts
        pts = case["problems"] * (case["points"] - 16) / math.log(case["points"] / 16)
        walks = pts * (case["walks"] - 64) / math.log(case["walks"] / 64)
        read = case["problems"] * 4 * 64 * 64 * 4 + pts * 12
    else:
        pts = case["points"] ** 2 if kind == "slice" else case["points"]
        walks = pts * case["walks"]
        read = pts * (8 if p in DIM2 else 12)
        if p in ("mesh", "mesh_manufactured"):
            read += 20 * 4 ** case["level"] * (12 + 6) + (3 * 128 ** 3 * 4 if p == "mesh" else 0)
        if kind == "inverse":
            read += 4 * (32 ** 3 + 16 ** 3)
    written = pts * 8 * {"host": 3, "grad": 4 + 3 * (2 if p in DIM2 else 3), "inverse": 1, "slice": 3}.get(kind, 4)
    if kind == "slice":
        read, written = read + pts * 24, written + 4 * case["width"] * case["height"]
    if kind == "inverse":
        written += 4 * (32 ** 3 + 16 ** 3)
    # the inverse step needs the walks once and their scatter (128 taps of two grids); the series next-flight
    # ball costs a sweep of its terms on top of the step
    per = FLOPS[p] + {"inverse": 900.0, "nf": 60.0 * case.get("terms", 0) + 200.0}.get(kind, 0.0)
    return {"bytes": float(read + written), "flops": float(walks * STEPS[p] * per)}


# ---- the same walks in 64 bits (plain torch), for the two manufactured box problems ----
def _philox(c, seed):
    m = 0xFFFFFFFF

    def hilo(a, b):  # 32 x 32 -> 64 bits without leaving int64
        t = (b & 0xFFFF) * a
        u = (b >> 16) * a + (t >> 16)
        return u >> 16, ((u & 0xFFFF) << 16) | (t & 0xFFFF)
    k0, k1 = seed & m, (seed >> 32) & m
    x, y, z, w = c
    for _ in range(10):
        h0, l0 = hilo(0xD2511F53, x)
        h1, l1 = hilo(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return x, y, z, w


def _fields(problem, x):
    """sigma', f', gamma and the boundary data u at x [dim, n], in closed form (u, alpha, sigma, Phi of the two
    problems, differentiated by hand)."""
    pi, s, c = math.pi, torch.sin, torch.cos
    zero = torch.zeros_like(x[0])
    if problem == "square2d":
        X, Y = x[0], x[1]
        u = s(pi * X) * torch.cosh(Y)
        gu, lu = (pi * c(pi * X) * torch.cosh(Y), s(pi * X) * torch.sinh(Y)), (1 - pi * pi) * u
        al = 1 + 0.5 * s(2 * pi * X) * c(2 * pi * Y)
        ga = (pi * c(2 * pi * X) * c(2 * pi * Y), -pi * s(2 * pi * X) * s(2 * pi * Y))
        la = -8 * pi * pi * (al - 1)
        sg, ph, gp, lp = 2 + s(3 * X + Y), zero, (zero, zero), zero
    else:
        X, Y, Z = x[0], x[1], x[2]
        e = torch.exp(0.5 * X)
        u = e * s(pi * Y) * c(pi * Z)
        gu = (0.5 * u, pi * e * c(pi * Y) * c(pi * Z), -pi * e * s(pi * Y) * s(pi * Z))
        lu = (0.25 - 2 * pi * pi) * u
        al, la = 1 + 0.3 * (X * X + Y * Y + Z * Z), zero + 1.8
        ga = (0.6 * X, 0.6 * Y, 0.6 * Z)
        sg = 1 + X * Y
        ph = X * s(2 * pi * Y) + s(2 * pi * Z) / (2 * pi) + 0.5 * Z
        gp = (s(2 * pi * Y), 2 * pi * X * c(2 * pi * Y), c(2 * pi * Z) + 0.5)
        lp = -4 * pi * pi * X * s(2 * pi * Y) - 2 * pi * s(2 * pi * Z)
    f = -(al * lu + sum(a * b for a, b in zip(ga, gu))) - al * sum(a * b for a, b in zip(gp, gu)) + sg * u
    gg = [0.5 * (a / al + p) for a, p in zip(ga, gp)]
    lg = 0.5 * (la / al - sum(a * a for a in ga) / al ** 2 + lp)
    gam = 0.5 * torch.log(al) + 0.5 * ph
    return sg / al + lg + sum(a * a for a in gg), torch.exp(gam) * f / al, gam, u


def _tail_sinh(y):  # sinh y - y
    t = y * y
    ser = torch.zeros_like(y)
    for k in range(12, 0, -1):
        ser = (1 + ser) * t / ((2 * k) * (2 * k + 1))
    return torch.where(y < 1, y * ser, torch.sinh(y) - y)


def _green(dim, a):
    """sigma_bar |G| of the centred ball with a = sqrt(sigma_bar) R."""
    if dim == 3:
        return _tail_sinh(a) / torch.sinh(a)
    t, ser = 0.25 * a * a, torch.zeros_like(a)
    for k in range(25, 0, -1):
        ser = (1 + ser) * t / (k * k)
    return torch.where(a < 4, ser / (1 + ser), 1 - 1 / torch.special.i0(a))


def _radius(dim, a, u):
    """rho = r/R with the radial cumulative distribution of G/|G| equal to u, by bisection."""
    lo, hi = torch.zeros_like(a), torch.ones_like(a)
    sp = torch.special
    if dim == 3:
        sa = _tail_sinh(a)
    else:
        kr, norm = sp.modified_bessel_k0(a) / sp.i0(a), _green(2, a)
    for _ in range(48):
        r = 0.5 * (lo + hi)
        t = a * r
        if dim == 3:
            y = a - t
            F = 1 - (_tail_sinh(y) + 2 * t * torch.sinh(0.5 * y) ** 2) / sa
        else:
            F = (1 - t * sp.modified_bessel_k1(t) - kr * t * sp.i1(t)) / norm
        up = F < u
        lo, hi = torch.where(up, r, lo), torch.where(up, hi, r)
    return 0.5 * (lo + hi)


def _sigma_bar(problem, dim, m):
    c = (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m
    sp = _fields(problem, torch.stack([g.reshape(-1) for g in torch.meshgrid(*([c] * dim), indexing="ij")]))[0]
    return max(float(sp.max() - sp.min()), float(sp.max()), 1e-3 / dim)


def exact(case, seed):
    problem, dim = case["problem"], 2 if case["problem"] in DIM2 else 3
    if case["kind"] not in ("solve", "host") or problem not in ("square2d", "cube3d") or \
            case["points"] * case["walks"] > (1_000_000 if dim == 2 else 2_500_000):
        return None
    npts, walks, eps = case["points"], case["walks"], EPS.get(problem, 1e-4)
    sb = _sigma_bar(problem, dim, LATTICE.get(problem, 64))
    root = math.sqrt(sb)
    x0 = torch.from_numpy(_points(case, seed)).cuda().double()
    item = torch.arange(npts * walks, device="cuda")
    p, w = item // walks, item % walks
    x = x0[:, p]
    val = torch.zeros(npts * walks, dtype=torch.float64, device="cuda")
    W_, acc, k = torch.ones_like(val), torch.zeros_like(val), 0
    turn = 2 * math.pi
    while item.numel():
        near = torch.stack([x, 1 - x]).reshape(2 * dim, -1)
        d, side = near.min(0)
        end = ~(d >= eps)
        if bool(end.any()):
            xe = x[:, end]
            xb, ax = xe.clone(), side[end]
            xb[ax % dim, torch.arange(ax.numel(), device="cuda")] = (ax >= dim).double()
            val[item[end]] = acc[end] + W_[end] * torch.exp(_fields(problem, xe)[2]) * _fields(problem, xb)[3]
            go = ~end
            item, p, w, x, W_, acc, d = item[go], p[go], w[go], x[:, go], W_[go], acc[go], d[go]
        if not item.numel():
            break
        c = _philox((p, w, torch.full_like(p, k), torch.zeros_like(p)), int(seed))
        if dim == 2:
            mu, ur, ty, tz = (((v >> 9).double() + 0.5) * 2.0 ** -23 for v in c)
            dy, dz = (torch.stack([torch.cos(turn * t), torch.sin(turn * t)]) for t in (ty, tz))
        else:
            low = [((c[i] & 0x7FF) << 10) | (c[i + 2] & 0x3FF) for i in (0, 1)]
            mu, ur, cy, fy, cz, fz = ((v.double() + 0.5) * 2.0 ** -21 for v in [v >> 11 for v in c] + low)

            def direction(cu, fu):
                cs = 1 - 2 * cu
                sn = torch.sqrt(torch.clamp(1 - cs * cs, min=0))
                return torch.stack([sn * torch.cos(turn * fu), sn * torch.sin(turn * fu), cs])
            dy, dz = direction(cy, fy), direction(cz, fz)
        a = root * d
        pb = _green(dim, a)
        y = x + d * _radius(dim, a, ur) * dy
        sp, fp, _, _ = _fields(problem, y)
        acc = acc + W_ * (pb / sb) * fp
        null = mu <= pb
        W_ = torch.where(null, W_ * (1 - sp / sb), W_)
        x = torch.where(null, y, x + d * dz)
        k += 1
    u = val.reshape(npts, walks) * torch.exp(-_fields(problem, x0)[2])[:, None]
    mean = u.mean(1)
    var = u.var(1) if walks > 1 else torch.zeros_like(mean)
    out = [mean, var, torch.sqrt(var / walks)]
    return out if case["kind"] == "host" else out + [None]
