"""The two-level preconditioner's monopole sums over a cluster tree (2,048
panels and more) and directly (one panel fewer), against the definition
written out with numpy: at the switch, with a full and with a short last
cluster."""
import numpy as np
import pytest

from dc_synth.drawings import make_closed_set
from test_gpu_precond import reference_M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("curves,per_curve", [(23, 89), (16, 128), (13, 159)])   # 2047, 2048, 2067 panels
def test_cluster_preconditioner_matches_definition(dcmod, cuda_ok, oracle_mod, curves, per_curve):
    # Bound: the coarse inverse is FP32 with an inverse_check below 1e-3 by
    # its own acceptance; the cluster sums add 0.4^9 / 9 = 3e-5 of a far term.
    import torch
    d = make_closed_set(61, n_curves=curves, panels_per_curve=per_curve, g=4)
    assert d.n_panels == curves * per_curve
    ctx = dcmod.Context(form="fmm32", g=d.g, s_per_panel=d.s_per_panel, p=24, leaf_size=32)
    ctx.build_drawing(d)
    info = ctx.precond_info()
    assert info["two_level"] == 1.0 and info["panels"] == d.n_panels
    M, N = reference_M(oracle_mod, d)
    v = np.random.default_rng(53).standard_normal((N, 3))
    got = torch.empty((N, 3), dtype=torch.float64, device="cuda")
    ctx.apply_operator(torch.from_numpy(v).cuda(), got, 0, 3)
    torch.cuda.synchronize()
    ref = M(v)
    rel = np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref)
    print(f"{d.n_panels} panels: relative difference to the definition {rel:.2e}")
    assert rel < 1e-3
