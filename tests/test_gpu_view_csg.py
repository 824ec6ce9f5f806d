"""The sphere-traced view of CSG lists, whose steps are decided in FP32 where that suffices, against
the same tracing in numpy (FP64 throughout)."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _prim(prim, p, x):
    p = np.asarray(p)
    if prim == "sphere":
        return np.linalg.norm(x - p[:3], axis=1) - p[3]
    if prim == "box":
        q = np.abs(x - p[:3]) - (p[3:6] - p[6])
        out = np.linalg.norm(np.maximum(q, 0), axis=1)
        return np.where(out > 0, out, q.max(1)) - p[6]
    if prim == "capsule":
        ab, ax = p[3:6] - p[:3], x - p[:3]
        t = np.clip(ax @ ab / (ab @ ab), 0, 1)
        return np.linalg.norm(ax - t[:, None] * ab, axis=1) - p[6]
    if prim == "torus":
        v = x - p[:3]
        return np.hypot(np.hypot(v[:, 0], v[:, 1]) - p[3], v[:, 2]) - p[4]
    return (x - p[:3]) @ p[3:6]


def _sdf(nodes, x):
    d = None
    for prim, op, p in nodes:
        s = _prim(prim, p, x)
        if d is None:
            d = s
        elif op == "union":
            d = np.minimum(d, s)
        else:
            d = np.maximum(d, -s if op == "subtract" else s)
    return d


SPHERE = ("sphere", "union", [0.0, 0.0, 0.0, 0.8])
SCENES = {
    "scene": W.csg_scene_3d(),
    # the same sphere twice: FP32 never tells which of the two decides
    "tie": W.csg([-1, -1, -1], [1, 1, 1], SPHERE, SPHERE),
    # a crease in the view's plane of symmetry, a half-space with a long normal, a huge cut
    "crease": W.csg([-1.3, -1, -1], [1.3, 1, 1], ("sphere", "union", [-0.4, 0, 0, 0.8]), ("sphere", "union", [0.4, 0, 0, 0.8]),
                    ("halfspace", "intersect", [0, -0.5, 0, 0, -7.0, 0]), ("sphere", "subtract", [0, 80.0, 0, 79.4])),
    "sixteen": W.csg([-1, -1, -1], [1, 1, 1], *[("sphere", "union" if i % 3 else "subtract",
                                                 [0.6 * math.cos(i), 0.6 * math.sin(i), 0.1 * (i % 5 - 2), 0.3])
                                                if i else SPHERE for i in range(16)]),
}


@pytest.mark.parametrize("name", list(SCENES))
@pytest.mark.parametrize("w,h", [(96, 64), (33, 31)])
def test_depth_equals_fp64_tracing(name, w, h):
    """A ray stops within tol = 1e-5 of the box diagonal; the two tracings round differently, so
    their depths agree to 2 tol except on rays that graze the surface (a step more or less
    there: at most 1 % of the pixels)."""
    import torch

    import paper_2201_13240_gb300 as wos
    dom = SCENES[name]
    u = W.sst(W.term(1.0, (W.LIN, 1.0, 0.0)))
    prob_desc = W.problem(3, dom, W.const(1.0), W.zero(), W.zero(), u, um=u)
    ctx = wos.Context(0)
    prob = ctx.problem(prob_desc)
    eye, n = np.array([0.0, 0.4, 4.0]), 16
    v = wos.view([-1.3, -1.3, 0.2], [2.6, 0, 0], [0, 2.6, 0], n, n, w, h, (-1.0, 1.0), eye=tuple(eye))
    acc = ctx.new_accum(n * n)
    acc[2].fill_(1)
    _, val, dep = ctx.render_slice(prob, v, acc, with_value=True, with_depth=True)
    dep, val = dep.cpu().numpy().reshape(-1), val.cpu().numpy().reshape(-1)

    fwd = -eye / np.linalg.norm(eye)
    right = np.cross(fwd, [0, 1, 0])
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    th = math.tan(math.radians(40.0) / 2)
    px, py = np.meshgrid(np.arange(w), np.arange(h))
    sx = ((px.reshape(-1) + 0.5) / w * 2 - 1) * th * w / h
    sy = (1 - (py.reshape(-1) + 0.5) / h * 2) * th
    d = fwd + sx[:, None] * right + sy[:, None] * up
    d /= np.linalg.norm(d, axis=1)[:, None]
    p = np.array(dom["p"])
    scale = np.linalg.norm(p[3:6] - p[:3])
    tol = 1e-5 * scale
    t, want, plane = np.zeros(w * h), np.full(w * h, np.inf), np.zeros(w * h, bool)
    live = np.ones(w * h, bool)
    for _ in range(512):
        x = eye + t[:, None] * d
        sd, sp = _sdf(dom["nodes"], x), x[:, 2] - 0.2
        s = np.maximum(sd, sp)
        hit = live & (s < tol)
        want[hit], plane[hit] = t[hit], (sp >= sd)[hit]
        live &= ~hit
        t = np.where(live, t + np.maximum(s, tol), t)
        live &= t < 1e3 * scale
        if not live.any():
            break
    same = np.isfinite(dep) == np.isfinite(want)
    close = same & (~np.isfinite(want) | (np.abs(np.where(np.isfinite(want), dep - want, 0)) <= 2 * tol))
    assert close.mean() >= 0.99, close.mean()
    assert np.isfinite(want).mean() > 0.05
    # pixels of the slice plane show its (zero) mean, the others none
    a, b = (x[:, 0] + 1.3) / 2.6, (x[:, 1] + 1.3) / 2.6
    shown = plane & np.isfinite(want) & (a >= 0) & (a < 1) & (b >= 0) & (b < 1)
    assert (np.isfinite(val) == shown).mean() >= 0.99
