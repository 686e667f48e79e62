"""The FP64 forms' float-float pixels and coefficients where their frames are
strained: targets 1e-16 to 1e-12 off a curve while the frame is as wide as
the canvas, canvases far outside the float range of a squared distance, and
leaves that stop at the depth limit with thousands of pieces.  Tolerance:
1e-11 of the field, the FP64 forms' own."""
import dataclasses

import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values
from dc_synth.drawings import Drawing
from test_gpu_render_frames import _render, library_discretisation, line_distance

pytestmark = pytest.mark.gpu


def _lines(seed, n, g=4):
    """Long straight curves across the page, one panel each."""
    rng = np.random.default_rng(seed)
    a, b = rng.uniform(0.05, 0.4, (n, 2)), rng.uniform(0.6, 0.95, (n, 2))
    flip = rng.uniform(size=n) < 0.5
    a[flip, 0], b[flip, 0] = 1.0 - a[flip, 0], 1.0 - b[flip, 0]
    t = np.arange(4)[None, :, None] / 3.0
    ctrl = (1 - t) * a[:, None] + t * b[:, None]
    return Drawing("lines", ctrl, np.zeros(n, bool), rng.uniform(0, 1, (n, 2, 2, 3)), np.arange(n + 1, dtype=np.int32),
                   np.zeros(n), g=g, s_per_panel=5 * g)


@pytest.mark.parametrize("form,leaf", [("dense64", 64), ("fmm64", 4096), ("fmm64", 8)])
def test_side_of_a_long_segment(dcmod, cuda_ok, oracle_mod, form, leaf):
    O = oracle_mod
    d = _lines(3, 6)
    disc = library_discretisation(dcmod, O, d)
    up, um = O.boundary_values(d, disc)
    sig = random_node_values(disc.n_nodes, seed=41)
    ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, p=30, leaf_size=leaf,
                        domain=(-1.0, -1.0, 2.0, 2.0))
    ctx.build_drawing(d)
    ctx.set_density(sig)
    # a row of 64 pixels across the page, one of them a few units in the last
    # place off a segment; steps of 1/64 from a multiple of 2^-52 are exact
    rng = np.random.default_rng(42)
    views, hits = [], []
    for _ in range(600):
        k, t, c = rng.integers(disc.n_segments), rng.uniform(0.2, 0.8), int(rng.integers(64))
        x1, y1, x2, y2 = disc.seg_xy[k]
        off = rng.choice([-1, 1]) * np.exp(rng.uniform(np.log(1e-16), np.log(1e-12)))
        n = np.array([y2 - y1, x1 - x2]) / np.hypot(x2 - x1, y2 - y1)
        q = np.array([x1 + t * (x2 - x1), y1 + t * (y2 - y1)]) + off * n
        grid = lambda v: np.round(v * 2.0 ** 52) / 2.0 ** 52
        x0, y0 = grid(q[0] - (c + 0.5) / 64), grid(q[1] - 0.5 / 64)
        views.append((x0, y0, x0 + 1.0, y0 + 1.0 / 64, 64, 1))
        hits.append(64 * len(hits) + c)
    got = _render(dcmod, ctx, views)
    pts = np.concatenate([O.pixel_centres(v[:4], v[4], v[5]) for v in views])
    ref = O.layer_potential(disc, pts, sig, up - um)
    dist = line_distance(disc.seg_xy, pts[hits])
    keep = np.ones(len(pts), bool)
    keep[np.array(hits)[dist < 5e-17]] = False
    assert (dist < 2e-12).all() and (dist < 1e-15).sum() > 50
    assert np.abs(got - ref)[keep].max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("form", ["dense64", "fmm64"])
@pytest.mark.parametrize("e", [-60, -50, -45, -9, 0, 21, 62, 66, 80])
def test_canvas_outside_the_float_range(dcmod, cuda_ok, oracle_mod, form, e):
    O = oracle_mod
    s = 2.0 ** e
    d = drawing_by_name("closed4")
    d = dataclasses.replace(d, ctrl=d.ctrl * s)
    disc = library_discretisation(dcmod, O, d)
    up, um = O.boundary_values(d, disc)
    sig = random_node_values(disc.n_nodes, seed=43, scale=1.0 / s)
    ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, p=30, domain=(0.0, 0.0, s, s))
    ctx.build_drawing(d)
    ctx.set_density(sig)
    views = [(0.0, 0.0, s, s, 65, 31), (0.3 * s, 0.4 * s, 0.301 * s, 0.401 * s, 20, 20)]
    got = _render(dcmod, ctx, views)
    pts = np.concatenate([O.pixel_centres(v[:4], v[4], v[5]) for v in views])
    ref = O.layer_potential(disc, pts, sig, up - um)
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("depth", [1, 2, 40])
def test_operator_with_leaves_at_the_depth_limit(dcmod, cuda_ok, oracle_mod, depth):
    import torch
    d = drawing_by_name("mixed16")
    disc = library_discretisation(dcmod, oracle_mod, d)
    rows = oracle_mod.hybrid_rows(disc)
    ctx = dcmod.Context(form="fmm64", g=d.g, s_per_panel=d.s_per_panel, p=30, max_depth=depth, domain=(0.0, 0.0, 1.0, 1.0))
    ctx.build_drawing(d)
    v = random_node_values(disc.n_nodes, seed=71)
    x = torch.from_numpy(v).cuda()
    y = torch.empty_like(x)
    for op in (0, 1):
        ctx.apply_operator(x, y, op)
        torch.cuda.synchronize()
        ref = rows[op] @ v
        err = np.abs(y.cpu().numpy() - ref).max() / np.abs(ref).max()
        print(f"depth {depth} op {op}: {err:.2e}")
        assert err <= 1e-11
