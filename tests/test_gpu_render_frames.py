"""The FP32 form's pixel rectangles where their frames are strained: canvases
far from the origin and in pixel units, where a pixel's side of a curve is
finer than the (hi, lo) coordinates; sources at the distance that decides
whether a rectangle samples them; rectangles so small that their radius
leaves the float range; channels of very different size; the mean of a large
far field.  Tolerance: the form's 1e-5 of the field where none is derived.
"""
import dataclasses

import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values
from dc_synth.drawings import Drawing

pytestmark = pytest.mark.gpu

DOMAIN = (-0.5, -0.5, 1.5, 1.5)


def _render(dcmod, ctx, views):
    import torch
    out = torch.empty((sum(v[4] * v[5] for v in views), 3), dtype=torch.float64, device="cuda")
    ctx.render_viewport(views, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def library_discretisation(dcmod, O, d):
    """The oracle's discretisation with the library's own end points, which
    differ from it by some 1e-13."""
    disc = O.discretise(d)
    own = dcmod.aux_discretise(d.ctrl, d.panel_ptr, d.panel_start, d.colours, d.g, d.s_per_panel)
    return dataclasses.replace(disc, node_xy=own["node_xy"], seg_xy=own["seg_xy"], seg_w=own["seg_w"])


def line_distance(seg, pts):
    """Distances of pts from the nearest of the segments, in extended precision."""
    q = np.asarray(pts, np.longdouble)[:, None]
    a, b = np.asarray(seg[:, :2], np.longdouble)[None], np.asarray(seg[:, 2:], np.longdouble)[None]
    ab = b - a
    t = np.clip(((q - a) * ab).sum(2) / (ab * ab).sum(2), 0, 1)
    e = a + t[..., None] * ab - q
    return np.sqrt((e * e).sum(2)).min(1).astype(float)


@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (2048.0, 0.0), (2.0 ** 16, 0.0), (1.0, 300.0), (64.0, -5000.0)])
def test_side_of_a_curve_far_from_the_origin(dcmod, cuda_ok, oracle_mod, scale, shift):
    O = oracle_mod
    d = drawing_by_name("mixed16")
    d = dataclasses.replace(d, ctrl=d.ctrl * scale + shift)
    disc = library_discretisation(dcmod, O, d)
    up, um = O.boundary_values(d, disc)
    sig = random_node_values(disc.n_nodes, seed=35, scale=1.0 / scale)
    ctx = dcmod.Context(form="fmm32", g=d.g, s_per_panel=d.s_per_panel, p=24,
                        domain=tuple(shift + scale * c for c in DOMAIN))
    ctx.build_drawing(d)
    ctx.set_density(sig)
    big = np.abs(disc.seg_xy).max()
    ulp = 2.0 ** (np.floor(np.log2(big)) - 52)
    views = []
    for k in range(5, disc.n_segments, 211):
        x1, y1, x2, y2 = disc.seg_xy[k]
        mx, my = np.round(0.5 * (x1 + x2) / ulp) * ulp, np.round(0.5 * (y1 + y2) / ulp) * ulp
        for w, h, px in ((16, 16, 2 * ulp), (16, 16, 16 * ulp), (7, 6, 8 * ulp)):   # sampled and direct
            views.append((mx - w // 2 * px, my - h // 2 * px, mx + (w - w // 2) * px, my + (h - h // 2) * px, w, h))
    got = _render(dcmod, ctx, views)
    pts = np.concatenate([O.pixel_centres(v[:4], v[4], v[5]) for v in views])
    ref = O.layer_potential(disc, pts, sig, up - um)
    # 64-bit coordinates and products of them decide the side beyond a few units in the last place
    keep = np.concatenate([line_distance(disc.seg_xy[np.abs(disc.seg_xy[:, :2] - p[:1]).max(1) < 0.05 * scale], p)
                           for p in np.split(pts, np.cumsum([v[4] * v[5] for v in views])[:-1])]) > 4 * ulp
    assert keep.sum() > 0.3 * len(pts)
    assert np.abs(got - ref)[keep].max() <= 1e-5 * max(1.0, np.abs(ref).max())


def _spokes(centre, radii, length, angles, g=4):
    """Straight radial curves from the given radii outward, one panel each."""
    u = np.stack([np.cos(angles), np.sin(angles)], 1)
    a = centre + radii[:, None] * u
    ctrl = a[:, None] + (length * np.arange(4) / 3.0)[None, :, None] * u[:, None]
    n = len(angles)
    col = np.random.default_rng(5).uniform(0, 1, (n, 2, 2, 3))
    return Drawing("spokes", ctrl, np.zeros(n, bool), col, np.arange(n + 1, dtype=np.int32), np.zeros(n), g=g,
                   s_per_panel=5 * g)


@pytest.mark.parametrize("sep,scale,n", [(2.5, 3.0, 96), (2.5, 3.0, 10), (5.0, 3e4, 96)])
def test_sources_at_the_sampling_distance(dcmod, cuda_ok, sep, scale, n):
    # the rectangle of rows and columns 24 .. 31 of 64: radius 3.5 sqrt(2) pixels about its centre; near
    # ends at sep radii, off by a few units in the last place of the floats that are compared
    dx = 1.0 / 64
    centre = np.array([28 * dx, 28 * dx])
    near = sep * 3.5 * np.sqrt(2.0) * dx
    radii = near * (1.0 + (np.arange(n) % 33 - 16) * 2.0 ** -24)
    d = _spokes(centre, radii, 4 * dx, 0.1 + 2 * np.pi * np.arange(n) / n)
    got, sig = {}, random_node_values(d.n_nodes, seed=36, scale=scale)
    for form in ("fmm32", "fmm64"):
        ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, leaf_size=4096, domain=(0.0, 0.0, 1.0, 1.0))
        ctx.build_drawing(d)
        ctx.set_density(sig)
        got[form] = _render(dcmod, ctx, [(0.0, 0.0, 1.0, 1.0, 64, 64)])
        ctx.close()
    assert np.abs(got["fmm32"] - got["fmm64"]).max() <= 1e-5 * max(1.0, np.abs(got["fmm64"]).max())


@pytest.mark.parametrize("scale", [3.0, 3000.0])   # 3000: large sources, whose polynomial is in FP64
@pytest.mark.parametrize("size", [1e-18, 1e-21, 1e-24, 1e-30, 1e-44, 1e-60, 1e-300])
def test_rectangles_below_the_float_range(dcmod, cuda_ok, size, scale):
    d = drawing_by_name("mixed16")
    views = [(0.0, 0.0, size, size, 64, 64), (0.0, 0.0, size, 0.5, 64, 9), (0.0, 0.0, 0.4, size, 50, 50),
             (-size, -size, size, size, 5, 5)]
    got, sig = {}, None
    for form in ("fmm32", "fmm64"):
        ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, domain=DOMAIN)
        ctx.build_drawing(d)
        if sig is None:
            sig = random_node_values(ctx.sizes().n_nodes, seed=37, scale=scale)
        ctx.set_density(sig)
        got[form] = _render(dcmod, ctx, views)
        ctx.close()
    assert np.isfinite(got["fmm64"]).all()
    assert np.abs(got["fmm32"] - got["fmm64"]).max() <= 1e-5 * max(1.0, np.abs(got["fmm64"]).max())


@pytest.mark.parametrize("channel", [0, 2])
def test_channel_beside_a_large_constant_one(dcmod, cuda_ok, channel):
    # a channel that is 5 inside the closed curves and 0 outside beside one a million times smaller: what the
    # small one loses has to be small against itself, so it is compared with its values when it is alone
    d = drawing_by_name("closed4")
    u, n = [], d.n_nodes
    sig = np.zeros((n, 3))
    sig[:, channel] = 1e-6 * random_node_values(n, seed=38)[:, 0]
    for jump in (5.0, 0.0):
        col = np.zeros_like(d.colours)
        col[:, 0, :, 1] = jump
        ctx = dcmod.Context(form="fmm32", g=d.g, s_per_panel=d.s_per_panel, domain=DOMAIN)
        ctx.build_drawing(dataclasses.replace(d, colours=col))
        ctx.set_density(sig)
        u.append(_render(dcmod, ctx, [(0.0, 0.0, 1.0, 1.0, 300, 200), (0.3, 0.3, 0.31, 0.32, 128, 96),
                                      (0.0, 0.0, 1.0, 1.0, 1100, 900)])[:, channel])
        ctx.close()
    assert np.abs(u[0] - u[1]).max() <= 1e-6 * np.abs(u[1]).max()


@pytest.mark.parametrize("views", [[(0.0, 0.0, 1.0, 1.0, 1100, 900)], [(0.0, 0.0, 1.0, 1.0, 311, 287)],
                                   [(x / 64, y / 64, (x + 1) / 64, (y + 1) / 64, 6, 7) for x in range(64) for y in range(64)]])
def test_large_far_field_is_not_biased(dcmod, cuda_ok, views):
    # 5 inside closed curves, nearly all of it from the expansions.  They are FP32, so a pixel is off by some
    # 1e-7 of its value and a leaf's mean by 2e-8 (its leading coefficient's rounding); a mean over a hundred
    # leaves and tens of thousands of pixels is not off by more than a few 1e-9
    d = drawing_by_name("closed4")
    col = np.zeros_like(d.colours)
    col[:, 1] = 5.0
    got, sig = {}, random_node_values(d.n_nodes, seed=39)
    for form in ("fmm32", "fmm64"):
        ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, leaf_size=16, domain=DOMAIN)
        ctx.build_drawing(dataclasses.replace(d, colours=col))
        ctx.set_density(sig)
        got[form] = _render(dcmod, ctx, views)
        ctx.close()
    big = np.abs(got["fmm64"]) > 3.0
    assert big.sum() > 10000
    mean = (got["fmm32"] / got["fmm64"] - 1.0)[big].mean()
    print(f"mean relative error {mean:.2e} of {big.sum()}")
    assert abs(mean) <= 1.5e-8
