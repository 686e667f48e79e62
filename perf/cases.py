"""What the speed of this library is measured on.

Each case is one pass through the public entry points of
``paper_2311_14312_gb300`` as a program that draws diffusion curves calls
them: rendering a density it has (Alg. 4), the whole way from the curves to
the image, applying the layer operators, evaluating points, and one
training step of the warm-start network.  The drawings are seeded random
ones of the shape of the repository's own (mixed open and closed cubics of
uneven size, panels by the library's adaptive rule).

The images are returned as the floating values; the 8-bit image is a
rounding of the same values and is not returned beside them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2311_14312_gb300 as dc

DOMAIN = (-0.5, -0.5, 1.5, 1.5)   # every viewport below lies inside it
PAIRS_EXACT = 2.0e10              # target-segment pairs a direct 64-bit sum takes in a few seconds
NODES_EXACT = 9000                # unknowns of a direct 64-bit solve


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # a thumbnail of a small drawing: the launches and their gaps count
        dict(name="render_thumb", kind="render", form="fmm32", curves=16, g=8, width=64, height=64, views=1, zoom=1.0,
             aa=0),
        # the page: the benchmark's size of drawing and image
        dict(name="render_page", kind="render", form="fmm32", curves=200, g=16, width=2048, height=2048, views=1,
             zoom=1.0, aa=0),
        # many uneven viewports of a large drawing, up to deep zooms, in one call
        dict(name="render_views", kind="render", form="fmm32", curves=2000, g=16, width=2200, height=2200, views=24,
             zoom=1e6, aa=0),
        # an odd-sized window zoomed in, with anti-aliased edges
        dict(name="render_smooth", kind="render", form="fmm32", curves=200, g=16, width=1021, height=613, views=1,
             zoom=3.0, aa=2),
        # the plain 64-bit form's image of a medium drawing
        dict(name="render_plain", kind="render", form="fmm64", curves=48, g=16, width=517, height=509, views=1,
             zoom=1.0, aa=0),
        # colours at scattered points (probes, samples along strokes)
        dict(name="points", kind="points", form="fmm32", curves=200, g=16, points=100003),
        # the layer operators at the nodes in the plain form (the matrix-vector product of a solver)
        dict(name="operator", kind="operator", form="fmm64", curves=200, g=16, panels=8),
        # curves to image while a small drawing is edited: build, solve, render into host memory
        dict(name="edit_small", kind="draw", form="fmm32", curves=16, g=8, width=256, height=256, tol=1e-10),
        # curves to image for the page
        dict(name="edit_page", kind="draw", form="fmm32", curves=200, g=16, width=2048, height=2048, tol=1e-10),
        # solve and render of a large drawing that is built already
        dict(name="solve_large", kind="solve", form="fmm32", curves=1000, g=16, width=2048, height=2048, tol=1e-8),
        # the dense 64-bit form from the curves to a small image: four closed curves, as its configuration says
        dict(name="dense_page", kind="draw", form="dense64", curves=4, g=16, width=128, height=128, tol=1e-12),
        # one training step's loss and gradient of the warm-start network (384 - 256 - 256 - 256 - 16)
        dict(name="train", kind="train", g=16, hidden=256, batch=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "plain", "points", "operator", "draw", "draw", "solve", "dense",
                       "train"])
    g = rng.choice([4, 8, 16, 16])
    if kind == "render":
        return dict(kind="render", form="fmm32", curves=_log_int(rng, 6, 1500), g=g, width=_log_int(rng, 40, 2048),
                    height=_log_int(rng, 40, 2048), views=rng.choice([1, 1, 1, 3, 12]),
                    zoom=rng.choice([1.0, 1.0, 4.0, 300.0, 1e6]), aa=rng.choice([0, 0, 0, 1, 2]))
    if kind == "plain":
        return dict(kind="render", form="fmm64", curves=_log_int(rng, 6, 120), g=g, width=_log_int(rng, 40, 640),
                    height=_log_int(rng, 40, 640), views=1, zoom=rng.choice([1.0, 1.0, 5.0]), aa=0)
    if kind == "points":
        return dict(kind="points", form=rng.choice(["fmm32", "fmm32", "fmm64"]), curves=_log_int(rng, 6, 400), g=g,
                    points=_log_int(rng, 100, 300000))
    if kind == "operator":
        return dict(kind="operator", form="fmm64", curves=_log_int(rng, 6, 500), g=g,
                    panels=rng.choice([6, 8, 11]))
    if kind == "draw":
        return dict(kind="draw", form="fmm32", curves=_log_int(rng, 6, 300), g=g, width=_log_int(rng, 100, 2048),
                    height=_log_int(rng, 100, 2048), tol=1e-10)
    if kind == "solve":
        return dict(kind="solve", form="fmm32", curves=_log_int(rng, 60, 1000), g=16, width=_log_int(rng, 256, 2048),
                    height=_log_int(rng, 256, 2048), tol=1e-8)
    if kind == "dense":
        return dict(kind="draw", form="dense64", curves=rng.randint(2, 4), g=rng.choice([8, 16]),
                    width=_log_int(rng, 40, 128), height=_log_int(rng, 40, 128), tol=1e-12)
    return dict(kind="train", g=rng.choice([8, 16]), hidden=rng.choice([72, 128, 256]), batch=_log_int(rng, 64, 12000))


# ------------------------------------------------------------------ inputs --
def _cells(rng, n):
    """n rectangles of uneven size that tile [0.04, 0.96]^2 (random bisection)."""
    todo, out = [((0.04, 0.04, 0.96, 0.96), n)], []
    while todo:
        (x0, y0, x1, y1), k = todo.pop()
        if k == 1:
            out.append((x0, y0, x1, y1))
            continue
        a = k // 2
        f = float(np.clip(a / k + rng.uniform(-0.18, 0.18), 0.15, 0.85))
        if x1 - x0 > y1 - y0:
            m = x0 + f * (x1 - x0)
            todo += [((x0, y0, m, y1), a), ((m, y0, x1, y1), k - a)]
        else:
            m = y0 + f * (y1 - y0)
            todo += [((x0, y0, x1, m), a), ((x0, m, x1, y1), k - a)]
    return out


def _panels(ctrl, m=64, ratio=0.2, levels=8):
    """Panels bisected in arc length while one is longer than ratio times its
    distance to the nearest other curve (on m points a curve), at least two
    a curve: the repository's rule for such drawings."""
    n, t = ctrl.shape[0], np.linspace(0.0, 1.0, m)[None, :, None]
    c = ctrl[:, None]
    p = (1 - t) ** 3 * c[:, :, 0] + 3 * t * (1 - t) ** 2 * c[:, :, 1] + 3 * t * t * (1 - t) * c[:, :, 2] + t ** 3 * c[:, :, 3]
    arc = np.concatenate([np.zeros((n, 1)), np.cumsum(np.hypot(*np.moveaxis(np.diff(p, axis=1), 2, 0)), 1)], 1)
    q = torch.from_numpy(p.reshape(-1, 2)).to("cuda" if torch.cuda.is_available() else "cpu")
    near, step = [], max(1, int(2e8 / (m * m * n)))
    for i in range(0, n, step):
        r = q[i * m:(i + step) * m]
        d2 = ((r[:, :1] - q[None, :, 0]) ** 2 + (r[:, 1:] - q[None, :, 1]) ** 2).view(-1, n, m).amin(2)
        d2[torch.arange(r.shape[0], device=q.device), i + torch.arange(r.shape[0], device=q.device) // m] = math.inf
        near.append(d2.amin(1))
    near = torch.cat(near).sqrt().cpu().numpy().reshape(n, m)
    ptr, start = [0], []
    for i in range(n):
        frac, todo, got = arc[i] / arc[i, -1], [(0.0, 1.0, 0)], []
        while todo:
            a, b, k = todo.pop()
            lo, hi = max(np.searchsorted(frac, a) - 1, 0), np.searchsorted(frac, b, side="right") + 1
            if k < levels and (k == 0 or (b - a) * arc[i, -1] > ratio * near[i, lo:hi].min()):
                todo += [(0.5 * (a + b), b, k + 1), (a, 0.5 * (a + b), k + 1)]
            else:
                got.append(a)
        start += sorted(got)
        ptr.append(len(start))
    return np.array(ptr, np.int32), np.array(start)


def _drawing(case, seed):
    """Control points, colours and panels of a random drawing: one simple
    cubic in each rectangle, 60 % open.  The dense case has closed ones with
    16 even panels each; where outputs are values at the nodes, the panels
    are even too, so that their number is the case's."""
    rng = np.random.default_rng([int(seed), 2311])
    n = case["curves"]
    dense = case.get("form") == "dense64"
    ctrl = np.zeros((n, 4, 2))
    closed = np.zeros(n, bool)
    for i, (x0, y0, x1, y1) in enumerate(_cells(rng, n)):
        size = 0.5 * min(x1 - x0, y1 - y0) / 1.25 * math.exp(rng.uniform(math.log(0.45), math.log(0.97)))
        a = rng.uniform(0.0, 2.0 * math.pi)
        closed[i] = dense or rng.uniform() < 0.4
        if closed[i]:
            q = np.array([[0.0, -0.9], [rng.uniform(1.2, 1.9), 0.9], [-rng.uniform(1.2, 1.9), 0.9], [0.0, -0.9]])
        else:
            q = np.array([[-1.0, rng.uniform(-0.6, 0.6)], [-0.3, rng.uniform(-1.0, 1.0)],
                          [0.3, rng.uniform(-1.0, 1.0)], [1.0, rng.uniform(-0.6, 0.6)]])
        q = q if rng.uniform() < 0.5 else q[::-1]
        turn = np.array([[math.cos(a), math.sin(a)], [-math.sin(a), math.cos(a)]])
        ctrl[i] = np.array([0.5 * (x0 + x1), 0.5 * (y0 + y1)]) + size * (q @ turn)
        if closed[i]:
            ctrl[i, 3] = ctrl[i, 0]
    colours = rng.uniform(0.0, 1.0, (n, 2, 2, 3))
    even = 16 if dense else case.get("panels", 0)
    if even:
        ptr, start = np.arange(n + 1, dtype=np.int32) * even, np.tile(np.arange(even) / even, n)
    else:
        ptr, start = _panels(ctrl)
    return dict(ctrl=ctrl, closed=closed, colours=colours, ptr=ptr, start=start, g=case["g"])


def _gauss(n):
    return np.polynomial.legendre.leggauss(n)


def _node_values(d, seed):
    """A density of the shape a solve gives: smooth along each curve with the
    inverse-square-root growth at the ends of open ones, of the size of a
    colour over the curve's length, and no total charge."""
    rng = np.random.default_rng([int(seed), 4312])
    n, g, ptr = d["ctrl"].shape[0], d["g"], d["ptr"]
    x, w = _gauss(g)
    curve = np.repeat(np.arange(n), np.diff(ptr))
    end = np.append(d["start"][1:], 1.0)
    end[ptr[1:] - 1] = 1.0
    width = end - d["start"]
    tau = d["start"][:, None] + width[:, None] * (0.5 * (x + 1.0))[None]
    t, tw = _gauss(32)
    t = (0.5 * (t + 1.0))[None, :, None]
    c = d["ctrl"][:, None]
    v = 3 * ((1 - t) ** 2 * (c[:, :, 1] - c[:, :, 0]) + 2 * t * (1 - t) * (c[:, :, 2] - c[:, :, 1])
             + t * t * (c[:, :, 3] - c[:, :, 2]))
    length = 0.5 * (np.hypot(v[..., 0], v[..., 1]) * tw).sum(1)
    k = rng.normal(0.0, 1.0, (n, 4, 3))[curve][:, None]
    tt = tau[..., None]
    sig = 0.4 * k[:, :, 0] + k[:, :, 1] * np.cos(2 * np.pi * tt) + k[:, :, 2] * np.sin(2 * np.pi * tt)
    tip = np.where(d["closed"][curve][:, None, None], 0.0, k[:, :, 3] / np.sqrt(tt * (1 - tt) + 1e-4))
    sig = (sig + 0.3 * tip) / length[curve][:, None, None]
    ds = 0.5 * (width * length[curve])[:, None] * w[None]
    sig -= (sig * ds[..., None]).sum((0, 1)) / ds.sum()
    return sig.reshape(-1, 3)


def _viewports(case, d, seed):
    """Whole-page views at zoom 1; else windows around points of curves, at
    zooms up to the case's, of uneven size when there are several."""
    rng = np.random.default_rng([int(seed), 77])
    out = []
    for i in range(case.get("views", 1)):
        w, h, z = case["width"], case["height"], case.get("zoom", 1.0)
        if case.get("views", 1) > 1:
            f = math.exp(math.log(0.12) * ((0.618034 * i + 0.3) % 1.0))
            w, h, z = max(8, int(w * f)), max(8, int(h * f)), math.exp(rng.uniform(0.0, math.log(z)))
        if z <= 1.0:
            out.append((0.0, 0.0, 1.0, 1.0, w, h))
            continue
        t = rng.uniform(0.05, 0.95)
        c = d["ctrl"][rng.integers(d["ctrl"].shape[0])]
        p = (1 - t) ** 3 * c[0] + 3 * t * (1 - t) ** 2 * c[1] + 3 * t * t * (1 - t) * c[2] + t ** 3 * c[3]
        hx, hy = 0.5 / z, 0.5 / z * h / w
        s = min(1.0, 0.45 / hy)
        out.append((float(p[0] - hx * s), float(p[1] - hy * s), float(p[0] + hx * s), float(p[1] + hy * s), w, h))
    return out


def _points(case, d, seed):
    """Scattered points: half uniform over the page, half close to curves."""
    rng = np.random.default_rng([int(seed), 99])
    n = case["points"]
    t, k = rng.uniform(0.0, 1.0, (n, 1)), rng.integers(d["ctrl"].shape[0], size=n)
    c = d["ctrl"][k]
    p = (1 - t) ** 3 * c[:, 0] + 3 * t * (1 - t) ** 2 * c[:, 1] + 3 * t * t * (1 - t) * c[:, 2] + t ** 3 * c[:, 3]
    a, r = rng.uniform(0.0, 2 * np.pi, n), np.exp(rng.uniform(math.log(1e-4), math.log(2e-2), n))
    p = p + np.stack([r * np.cos(a), r * np.sin(a)], 1)
    u = rng.uniform(0.0, 1.0, (n, 2))
    return np.clip(np.where(rng.uniform(size=(n, 1)) < 0.5, p, u), -0.2, 1.2)


def _train_inputs(case, seed):
    """Features of the ranges the feature rows have (geometry in panel
    lengths, unit vectors, colours), targets as wide as densities, and
    weights as a few steps after their initialisation leave them."""
    rng = np.random.default_rng([int(seed), 256])
    g, h, b = case["g"], case["hidden"], case["batch"]
    n_in = 22 * g + 32
    x = rng.uniform(0.0, 1.0, (b, n_in))
    x[:, :4 * g] = rng.uniform(-1.0, 1.0, (b, 4 * g))
    x[:, -32:] = rng.normal(0.0, 2.0, (b, 32))
    params = []
    for i, o in ((n_in, h), (h, h), (h, h), (h, g)):
        params += [rng.normal(0.0, math.sqrt(2.0 / i), o * i), rng.normal(0.0, 0.02, o)]
    target = rng.standard_t(4, (b, g)) * 3.0
    f = np.float32
    return x.astype(f), np.concatenate(params).astype(f), target.astype(f)


def prepare(case, seed):
    if case["kind"] == "train":
        x, p, t = (torch.from_numpy(v).cuda() for v in _train_inputs(case, seed))
        n = (22 * case["g"] + 32, case["hidden"], case["g"])
        work = torch.empty(dc.mlp_workspace_floats(*n, case["batch"]), device="cuda")
        return dict(case=case, n=n, x=x, p=p, t=t, work=work, grad=torch.empty_like(p), loss=torch.empty(1, device="cuda"))
    d = _drawing(case, seed)
    opts = dict(form=case["form"], g=d["g"], s_per_panel=5 * d["g"], domain=DOMAIN, aa_levels=case.get("aa", 0))
    if "tol" in case:
        opts.update(gmres_tol=case["tol"], gmres_max_iter=3000)
    ctx = dc.Context(**opts)
    s = dict(case=case, d=d, ctx=ctx)
    if case["kind"] != "draw":
        ctx.build_tree(d["ctrl"], d["ptr"], d["start"], d["colours"])
    if case["kind"] in ("render", "points"):
        ctx.set_density(_node_values(d, seed))
    wide = case["form"] != "fmm32"
    real = torch.float64 if wide else torch.float32
    if case["kind"] == "points":
        s["xy"] = torch.from_numpy(_points(case, d, seed)).cuda()
        s["out"] = torch.empty((case["points"], 3), dtype=real, device="cuda")
    elif case["kind"] == "operator":
        s["x"] = torch.from_numpy(_node_values(d, seed)).cuda()
        s["mu"] = torch.from_numpy(np.random.default_rng([int(seed), 5]).uniform(-1, 1, s["x"].shape)).cuda()
        s["y"], s["f"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
    else:
        s["views"] = _viewports(case, d, seed)
        px = sum(v[4] * v[5] for v in s["views"])
        if case["kind"] == "draw":   # the image goes to pinned host memory
            s["image"] = torch.empty((px, 3), dtype=real, pin_memory=True)
            s["out"] = s["image"].numpy()
        else:
            s["out"] = torch.empty((px, 3), dtype=real, device="cuda")
    return s


# --------------------------------------------------------------------- run --
def run(s):
    kind = s["case"]["kind"]
    if kind == "train":
        dc.mlp_loss_grad(*s["n"], s["p"], s["x"], s["t"], s["grad"], s["loss"], s["work"])
        return dict(loss=s["loss"], grad=s["grad"])
    ctx, d = s["ctx"], s["d"]
    if kind == "points":
        return ctx.eval_points(s["xy"], s["out"])
    if kind == "operator":
        return dict(single=ctx.apply_operator(s["x"], s["y"], op=0), double=ctx.apply_operator(s["mu"], s["f"], op=1))
    if kind == "draw":
        ctx.build_tree(d["ctrl"], d["ptr"], d["start"], d["colours"])
    if kind in ("draw", "solve"):
        ctx.solve_density()
    ctx.render_viewport(s["views"], rgb=s["out"])
    return s["out"]


def _counts(case):
    """About 7.5 panels a curve come from the adaptive rule."""
    panels = case["curves"] * (16 if case["form"] == "dense64" else case.get("panels", 7.5))
    return panels * case["g"], panels * 5 * case["g"]


def work(case):
    """Bytes: inputs read and outputs written once.  Flops where the method
    itself is a dense one: the network's products (forward, and two backward
    but for the first layer's inputs) and the dense form's pairs (45 each)."""
    if case["kind"] == "train":
        g, h, b = case["g"], case["hidden"], case["batch"]
        n_in = 22 * g + 32
        mats, first = n_in * h + 2 * h * h + h * g, n_in * h
        return dict(bytes=4.0 * (b * (n_in + g) + 2 * mats), flops=2.0 * b * (3 * mats - first))
    nodes, segs = _counts(case)
    real = 4.0 if case["form"] == "fmm32" else 8.0
    if case["kind"] == "points":
        return dict(bytes=24.0 * nodes + case["points"] * (16.0 + 3 * real), flops=0.0)
    if case["kind"] == "operator":
        return dict(bytes=2 * 48.0 * nodes, flops=0.0)
    px = float(case["width"]) * case["height"]
    if case.get("views", 1) > 1:   # the mean of the squared log-uniform factor
        px *= case["views"] * (1 - 0.12 ** 2) / (2 * math.log(1 / 0.12))
    flops = 45.0 * (2 * nodes + px) * segs if case["form"] == "dense64" else 0.0
    return dict(bytes=24.0 * nodes + 3 * real * px, flops=flops)


# ------------------------------------------------------------------- exact --
def _speed(c, t):
    u = 1.0 - t
    v = 3 * (u * u * (c[..., 1, :] - c[..., 0, :]) + 2 * t * u * (c[..., 2, :] - c[..., 1, :])
             + t * t * (c[..., 3, :] - c[..., 2, :]))
    return np.hypot(v[..., 0], v[..., 1])


def _t_of_s(ctrl, curve, s, cum, m):
    """Bezier parameters at arc lengths s of the given curves (Newton on the
    arc length, from the table cum of the lengths at j / m)."""
    x, w = _gauss(20)
    j = np.clip((cum[curve] <= s[:, None]).sum(1) - 1, 0, m - 1)
    base, c, t0 = cum[curve, j], ctrl[curve], j / m
    t = t0 + (s - base) / np.maximum(cum[curve, j + 1] - base, 1e-300) / m
    for _ in range(7):
        q = t0[:, None] + (t - t0)[:, None] * (0.5 * (x + 1.0))
        arc = base + 0.5 * (t - t0) * (_speed(c[:, None], q[..., None]) * w).sum(1)
        t = np.clip(t - (arc - s) / _speed(c, t[:, None]), 0.0, 1.0)
    return t


def _discretise(d):
    """Nodes on the solve polyline, segments, weights, boundary colours and
    the interpolation from nodes to segments, in 64 bits."""
    ctrl, ptr, start, g = d["ctrl"], d["ptr"], d["start"], d["g"]
    s, n, m = 5 * d["g"], d["ctrl"].shape[0], 64
    x20, w20 = _gauss(20)
    tq = (np.arange(m)[:, None] + 0.5 * (x20 + 1.0)) / m
    part = (_speed(ctrl[:, None, None], tq[None, ..., None]) * w20).sum(-1) * 0.5 / m
    cum = np.concatenate([np.zeros((n, 1)), np.cumsum(part, 1)], 1)
    curve = np.repeat(np.arange(n), np.diff(ptr))
    end = np.append(start[1:], 1.0)
    end[ptr[1:] - 1] = 1.0
    sa, sb = start * cum[curve, -1], end * cum[curve, -1]

    def params(frac):   # [panels, k] parameters at fractions of each panel
        arc = sa[:, None] + (sb - sa)[:, None] * frac[None]
        t = _t_of_s(ctrl, np.repeat(curve, frac.size), arc.ravel(), cum, m).reshape(arc.shape)
        t = np.where((start[:, None] == 0.0) & (frac[None] == 0.0), 0.0, t)
        return np.where((end[:, None] == 1.0) & (frac[None] == 1.0), 1.0, t)

    t = params(np.arange(s + 1) / s)[..., None]
    c = ctrl[curve][:, None]
    v = (1 - t) ** 3 * c[:, :, 0] + 3 * t * (1 - t) ** 2 * c[:, :, 1] + 3 * t * t * (1 - t) * c[:, :, 2] + t ** 3 * c[:, :, 3]
    seg = np.concatenate([v[:, :-1], v[:, 1:]], -1)
    chord = np.hypot(seg[..., 2] - seg[..., 0], seg[..., 3] - seg[..., 1])
    weight = ((sb - sa) / s)[:, None] / chord
    x, _ = _gauss(g)
    pos = 0.5 * (x + 1.0) * s
    k = np.minimum(np.floor(pos).astype(int), s - 1)
    node = seg[:, k, :2] + (pos - k)[None, :, None] * (seg[:, k, 2:] - seg[:, k, :2])
    own = np.arange(len(curve))[:, None] * s + k[None]
    tn = params(0.5 * (x + 1.0))[..., None]
    col = d["colours"][curve]
    up = (1 - tn) * col[:, None, 0, 0] + tn * col[:, None, 0, 1]
    um = (1 - tn) * col[:, None, 1, 0] + tn * col[:, None, 1, 1]
    mid = -1.0 + (2.0 * np.arange(s) + 1.0) / s
    lam = np.polynomial.legendre.legvander(mid, g - 1) @ np.linalg.inv(np.polynomial.legendre.legvander(x, g - 1))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return dict(node=dev(node.reshape(-1, 2)), own=dev(own.ravel()), seg=dev(seg.reshape(-1, 4)), w=dev(weight.ravel()),
                up=dev(up.reshape(-1, 3)), um=dev(um.reshape(-1, 3)), lam=dev(lam), g=g, s=s)


def _to_segments(D, v):
    return torch.einsum("km,pmc->pkc", D["lam"], v.reshape(-1, D["g"], 3)).reshape(-1, 3)


def _pair_integrals(D, q, own=None):
    """int G and int F over every segment (columns) for the targets q (rows)."""
    x1, y1, x2, y2 = D["seg"].T
    ax, ay, bx, by = (p[None] - q[:, i:i + 1] for p, i in ((x1, 0), (y1, 1), (x2, 0), (y2, 1)))
    dx, dy = (x2 - x1)[None], (y2 - y1)[None]
    c = torch.sqrt(dx * dx + dy * dy)
    cr = ax * dy - ay * dx                      # = a x b
    phi = torch.atan2(cr, ax * bx + ay * by)
    if own is not None:
        phi[torch.arange(q.shape[0], device=q.device), own] = 0.0
    ra, rb = ax * ax + ay * ay, bx * bx + by * by
    lg = torch.xlogy((bx * dx + by * dy) / c, rb) - torch.xlogy((ax * dx + ay * dy) / c, ra)
    k = -D["w"][None] / (2 * math.pi)
    return k * (0.5 * lg - c + cr / c * phi), k * phi


def _potential(D, q, sig, mu, own=None):
    S, out = D["seg"].shape[0], torch.empty((q.shape[0], 3), dtype=torch.float64, device=q.device)
    step = max(1, int(3e7 / S))
    for i in range(0, q.shape[0], step):
        G, F = _pair_integrals(D, q[i:i + step], None if own is None else own[i:i + step])
        part = 0.0
        if sig is not None:
            part = part + G @ sig
        if mu is not None:
            part = part + F @ mu
        out[i:i + step] = part
    return out


def _solve(D):
    N, g, s = D["node"].shape[0], D["g"], D["s"]
    A, Fm, mu = [], [], D["up"] - D["um"]
    step = max(1, int(3e7 / D["seg"].shape[0]))
    for i in range(0, N, step):
        G, F = _pair_integrals(D, D["node"][i:i + step], D["own"][i:i + step])
        A.append((G.reshape(G.shape[0], -1, s) @ D["lam"]).reshape(G.shape[0], N))
        Fm.append((F.reshape(F.shape[0], -1, s) @ D["lam"]).reshape(F.shape[0], N) @ mu)
    b = 0.5 * (D["up"] + D["um"]) - torch.cat(Fm)
    return torch.linalg.solve(torch.cat(A), b)


def _exact_train(case, seed):
    x, p, t = (torch.from_numpy(v).cuda() for v in _train_inputs(case, seed))
    g, h = case["g"], case["hidden"]
    dims, mats, at = (22 * g + 32, h, h, h, g), [], 0
    for i, o in zip(dims[:-1], dims[1:]):
        W = p[at:at + o * i].reshape(o, i).to(torch.bfloat16).double().requires_grad_()   # read as BF16
        b = p[at + o * i:at + o * i + o].double().requires_grad_()
        mats += [W, b]
        at += o * i + o
    y = x.double()
    for k in range(4):
        y = y @ mats[2 * k].T + mats[2 * k + 1]
        y = torch.nn.functional.gelu(y) if k < 3 else y
    loss = ((y - t.double()) ** 2).mean()
    return dict(loss=loss.detach().reshape(1), grad=torch.cat([v.reshape(-1) for v in torch.autograd.grad(loss, mats)]))


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case.get("aa", 0):
        return None
    d = _drawing(case, seed)
    nodes = int(d["ptr"][-1]) * d["g"]
    segs = 5 * nodes
    if case["kind"] == "operator":
        if nodes * segs > PAIRS_EXACT:
            return None
        D = _discretise(d)
        x = torch.from_numpy(_node_values(d, seed)).cuda()
        mu = torch.from_numpy(np.random.default_rng([int(seed), 5]).uniform(-1, 1, tuple(x.shape))).cuda()
        return dict(single=_potential(D, D["node"], _to_segments(D, x), None, D["own"]),
                    double=_potential(D, D["node"], None, _to_segments(D, mu), D["own"]))
    if case["kind"] == "points":
        q = torch.from_numpy(_points(case, d, seed)).cuda()
    else:
        q = []
        if sum(v[4] * v[5] for v in _viewports(case, d, seed)) * segs > PAIRS_EXACT:
            return None
        for x0, y0, x1, y1, w, h in _viewports(case, d, seed):
            px = x0 + (torch.arange(w, dtype=torch.float64, device="cuda") + 0.5) * ((x1 - x0) / w)
            py = y0 + (torch.arange(h, dtype=torch.float64, device="cuda") + 0.5) * ((y1 - y0) / h)
            q.append(torch.stack([px[None].expand(h, w), py[:, None].expand(h, w)], -1).reshape(-1, 2))
        q = torch.cat(q)
    if q.shape[0] * segs > PAIRS_EXACT or (case["kind"] in ("draw", "solve") and nodes > NODES_EXACT):
        return None
    D = _discretise(d)
    sig = _solve(D) if case["kind"] in ("draw", "solve") else torch.from_numpy(_node_values(d, seed)).cuda()
    return _potential(D, q, _to_segments(D, sig), _to_segments(D, D["up"] - D["um"]))
