"""The stored near-field coefficients of the node operator, formed in
float-float, and in FP64 with leaves too large or on a canvas too small for
that, against the oracle's rows of G_H and F_H: leaves of a few pieces, at the
switch, and so large that all pairs are near.  Tolerance: 1e-11 of the result, the FP64 forms' own at order 30."""
import dataclasses

import numpy as np
import pytest

from dc_synth import drawing_by_name, random_node_values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -9])
@pytest.mark.parametrize("leaf", [5, 64, 256, 257, 4000])
def test_operator_matches_the_oracle(dcmod, cuda_ok, oracle_mod, leaf, scale):
    import torch
    d = drawing_by_name("mixed16")
    d = dataclasses.replace(d, ctrl=d.ctrl * scale)
    disc = oracle_mod.discretise(d)
    rows = oracle_mod.hybrid_rows(disc)
    ctx = dcmod.Context(form="fmm64", g=d.g, s_per_panel=d.s_per_panel, p=30, leaf_size=leaf,
                        domain=(0.0, 0.0, scale, scale))
    ctx.build_drawing(d)
    v = random_node_values(disc.n_nodes, seed=71)
    x = torch.from_numpy(v).cuda()
    y = torch.empty_like(x)
    for op in (0, 1):
        ctx.apply_operator(x, y, op)
        torch.cuda.synchronize()
        ref = rows[op] @ v
        err = np.abs(y.cpu().numpy() - ref).max() / np.abs(ref).max()
        print(f"leaf {leaf} scale {scale:g} op {op}: {err:.2e}")
        assert err <= 1e-11
