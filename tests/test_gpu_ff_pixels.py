"""The pixels of the dense and the FP64 FMM form, summed in float-float,
against the oracle's direct sum: odd sizes, runs that end inside a block,
pixels on segment end points and midpoints, deep zooms.  Tolerance: 1e-11 of
the field, the FP64 forms' own."""
import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values

pytestmark = pytest.mark.gpu

DOMAIN = (-0.5, -0.5, 1.5, 1.5)


def _views(disc):
    out = [(0.0, 0.0, 1.0, 1.0, w, h) for w, h in ((1, 1), (63, 1), (1, 65), (33, 31), (129, 2))]
    for k, zoom in ((3, 50.0), (101, 2e3), (300, 1e6)):
        x1, y1, x2, y2 = disc.seg_xy[k]
        h = 0.5 / zoom
        out.append((x1 - h, y1 - h, x1 + h, y1 + h, 17, 17))                     # centre pixel: an end point
        out.append((0.5 * (x1 + x2) - h, 0.5 * (y1 + y2) - h, 0.5 * (x1 + x2) + h, 0.5 * (y1 + y2) + 2 * h, 16, 19))
    return out


@pytest.mark.parametrize("form,leaf", [("dense64", 64), ("fmm64", 64), ("fmm64", 5), ("fmm64", 300)])
def test_pixels_match_the_oracle(dcmod, cuda_ok, oracle_mod, form, leaf):
    import torch
    O = oracle_mod
    d = drawing_by_name("mixed16")
    disc = O.discretise(d)
    up, um = O.boundary_values(d, disc)
    sig = random_node_values(disc.n_nodes, seed=33, scale=30.0)
    ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, leaf_size=leaf, p=30, domain=DOMAIN)
    ctx.build_drawing(d)
    ctx.set_density(sig)
    views = _views(disc)
    out = torch.empty((sum(v[4] * v[5] for v in views), 3), dtype=torch.float64, device="cuda")
    ctx.render_viewport(views, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    pts = np.concatenate([O.pixel_centres(v[:4], v[4], v[5]) for v in views])
    # the side of a curve is decided by rounding for targets on it: keep those off it by more
    seg = disc.seg_xy
    keep = np.ones(len(pts), bool)
    for i, p in enumerate(pts):
        a, b = seg[:, :2], seg[:, 2:]
        ab = b - a
        t = np.clip(((p - a) * ab).sum(1) / (ab * ab).sum(1), 0, 1)
        keep[i] = np.hypot(*(a + t[:, None] * ab - p).T).min() > 1e-13
    ref = O.layer_potential(disc, pts, sig, up - um)
    assert np.isfinite(got).all() and keep.sum() > 0.95 * len(pts)
    assert np.abs(got - ref)[keep].max() <= 1e-11 * np.abs(ref).max()
