"""The FP64 forms' float-float pixels on canvases far outside the float range
of a squared distance, against the oracle's direct sum.  Tolerance: 1e-11 of
the field, the FP64 forms' own."""
import dataclasses

import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values
from test_gpu_render_frames import _render, library_discretisation

pytestmark = pytest.mark.gpu


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
