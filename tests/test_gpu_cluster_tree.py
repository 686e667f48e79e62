"""The cluster tree of the preconditioner's monopole sums: the sums
themselves against the definition (the coarse solution, whose FP32 inverse
would hide them, is eliminated), and a node that coincides, in floats, with
the only panel of a cluster outside its own."""
import dataclasses

import numpy as np
import pytest

from dc_synth.drawings import Drawing, make_closed_set
from test_gpu_precond import INV4PI

pytestmark = pytest.mark.gpu


def _operators(O, d):
    """P - B A~ P and B of M v = P y + B (v - A~ P y) (test_gpu_precond), without the coarse inverse."""
    disc = O.discretise(d)
    AG, _ = O.hybrid_rows(disc)
    N, g, P = disc.n_nodes, disc.g, disc.n_panels
    xy = disc.node_xy.reshape(P, g, 2)
    cen = xy.mean(axis=1)
    seg = disc.seg_xy.reshape(P, disc.nseg, 4)
    plen = (disc.seg_w.reshape(P, -1) * np.hypot(seg[..., 2] - seg[..., 0], seg[..., 3] - seg[..., 1])).sum(1)
    near = np.linalg.norm(cen[:, None] - cen[None], axis=2) < 1.5 * (plen[:, None] + plen[None, :])
    dxy = (disc.node_xy.astype(np.float32)[:, None] - cen.astype(np.float32)[None]).astype(np.float64)
    mono = -float(INV4PI) * np.log(np.maximum((dxy * dxy).sum(2), 1e-30))
    AP = np.where(np.repeat(near, g, axis=0), AG.reshape(N, P, g).sum(axis=2), plen[None, :] * mono)
    B = np.stack([np.linalg.inv(AG[j * g:(j + 1) * g, j * g:(j + 1) * g]) for j in range(P)])
    apply_b = lambda x: np.einsum("pij,pjc->pic", B, x.reshape(P, g, -1)).reshape(N, -1)
    return np.repeat(np.eye(P), g, axis=0) - apply_b(AP), apply_b, N


def _apply(dcmod, d, v):
    import torch
    ctx = dcmod.Context(form="fmm32", g=d.g, s_per_panel=d.s_per_panel, p=24, leaf_size=32,
                        domain=(0.0, 0.0, float(d.ctrl[..., 0].max()), float(d.ctrl[..., 1].max())))
    ctx.build_drawing(d)
    info = ctx.precond_info()
    assert info["two_level"] == 1.0 and info["panels"] == d.n_panels
    got = torch.empty(v.shape, dtype=torch.float64, device="cuda")
    ctx.apply_operator(torch.from_numpy(v).cuda(), got, 0, 3)
    torch.cuda.synchronize()
    return got.cpu().numpy()


def _distance(dcmod, O, d):
    """How far M v is from (P - B A~ P) y + B v for the best y, relative to M v."""
    C, apply_b, N = _operators(O, d)
    v = np.random.default_rng(54).standard_normal((N, 3))
    w = _apply(dcmod, d, v)
    assert np.isfinite(w).all()
    rhs = w - apply_b(v)
    y = np.linalg.solve(C.T @ C, C.T @ rhs)
    y += np.linalg.solve(C.T @ C, C.T @ (rhs - C @ y))
    return np.linalg.norm(rhs - C @ y) / np.linalg.norm(w)


def _closed(curves, per_curve, scale):
    d = make_closed_set(61, n_curves=curves, panels_per_curve=per_curve, g=4)
    return dataclasses.replace(d, ctrl=d.ctrl * scale)


@pytest.mark.parametrize("curves,per_curve,scale", [(16, 128, 1.0), (13, 159, 1.0),   # 2048, 2067 panels
                                                    (13, 159, 2.0 ** -34), (13, 159, 2.0 ** -56)])
def test_cluster_sums_match_definition(dcmod, cuda_ok, oracle_mod, curves, per_curve, scale):
    # Bound: as near as the direct sum, which takes over just below 2,048 panels, is on the same curves with
    # fewer panels, but for a factor of two (B enlarges the FP32 rounding of either; a separation of 1.5
    # instead of 2.5 would add terms that are off by 3e-3)
    O = oracle_mod
    rel = _distance(dcmod, O, _closed(curves, per_curve, scale))
    direct = _distance(dcmod, O, _closed(curves, 2047 // curves, scale))
    print(f"{curves * per_curve} panels, canvas {scale:g}: {rel:.2e}, direct {direct:.2e}")
    assert rel <= 2 * direct


def touching_drawing(fill=2040, gap=1e-9, g=4):
    """Straight one-panel curves: `fill` short ones in a grid, eight
    around the second to last centre and, alone in the last cluster, one
    whose centroid (0.9375, 0.9375) the last node of a long panel of the
    cluster before it misses by `gap`."""
    x = np.polynomial.legendre.leggauss(g)[0][-1]
    c, h = 0.9375, 0.02
    X = c - gap - x * h
    i = np.arange(fill)
    mid = [np.stack([0.02 + 0.01 * (i % 60), 0.02 + 0.01 * (i // 60)], 1)]
    half = [np.stack([0.003 * np.cos(i), 0.003 * np.sin(i)], 1)]
    k = np.arange(7)
    mid += [np.stack([X - 0.005 + 0.001 * k, np.full(7, c - 0.003)], 1), [[X, c]], [[c, c]]]
    half += [np.tile([[0.0, 0.0004]], (7, 1)), [[h, 0.0]], [[0.0, 0.001]]]
    mid, half = np.concatenate(mid), np.concatenate(half)
    t = (np.arange(4) * 2.0 / 3.0 - 1.0)[None, :, None]
    n = len(mid)
    return Drawing("touching", mid[:, None] + t * half[:, None], np.zeros(n, bool),
                   np.random.default_rng(6).uniform(0, 1, (n, 2, 2, 3)), np.arange(n + 1, dtype=np.int32), np.zeros(n),
                   g=g, s_per_panel=5 * g)


def test_node_on_the_centroid_of_another_cluster(dcmod, cuda_ok, oracle_mod):
    d, fewer = touching_drawing(), touching_drawing(fill=2032)
    assert d.n_panels % 8 == 1 and d.n_panels >= 2048 > fewer.n_panels
    assert _distance(dcmod, oracle_mod, d) <= 2 * _distance(dcmod, oracle_mod, fewer)
