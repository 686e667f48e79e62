"""The FP32 form's pixel rectangles (far field sampled on a circle, near
pieces per pixel) against the plain FP64 form on the same density: rectangle
edges and remainders, zooms at which the pieces are far longer than a
rectangle, leaves with more pieces than are staged at once, and densities
large enough for the FP64 terms.  Tolerance: the forms' 1e-5 colour
agreement, times the size of the field where that is larger than one."""
import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values

pytestmark = pytest.mark.gpu

DOMAIN = (-0.5, -0.5, 1.5, 1.5)


def _views(d):
    c = d.ctrl[3]
    p = (c[0] + 3 * c[1] + 3 * c[2] + c[3]) / 8          # a point of the curve
    out = [(0.0, 0.0, 1.0, 1.0, w, h) for w, h in ((1, 1), (7, 5), (48, 1), (8, 8), (9, 17), (64, 64), (129, 67),
                                                   (600, 511), (1030, 520))]
    for zoom, w, h in ((3.0, 200, 150), (40.0, 301, 100), (1e3, 130, 131), (1e5, 96, 64), (1e6, 700, 733)):
        out.append((p[0] - 0.5 / zoom, p[1] - 0.4 / zoom, p[0] + 0.5 / zoom, p[1] + 0.5 / zoom, w, h))
    return out


@pytest.mark.parametrize("leaf,scale", [(64, 3.0), (8, 3.0), (700, 3.0), (64, 3000.0), (700, 3000.0)])
def test_rectangles_match_the_plain_form(dcmod, cuda_ok, leaf, scale):
    import torch
    d = drawing_by_name("mixed16")
    sig = None
    got = {}
    for form in ("fmm32", "fmm64"):
        ctx = dcmod.Context(form=form, g=d.g, s_per_panel=d.s_per_panel, leaf_size=leaf, domain=DOMAIN)
        ctx.build_drawing(d)
        if sig is None:
            sig = random_node_values(ctx.sizes().n_nodes, seed=31, scale=scale)
        ctx.set_density(sig)
        views = _views(d)
        n = sum(v[4] * v[5] for v in views)
        rgb = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        ctx.render_viewport(views, rgb)
        torch.cuda.synchronize()
        got[form] = rgb.cpu().numpy()
        ctx.close()
    ref = got["fmm64"]
    assert np.isfinite(ref).all()
    tol = 1e-5 * np.maximum(1.0, np.abs(ref).max())
    assert np.abs(got["fmm32"] - ref).max() <= tol
