"""The warm-start network's tensor-core products at the edges of their tiles
(128 rows, 64 columns, 32 values of the sum) and of the ranges a weight
gradient's sum is cut into, aligned and not, against the FP64 oracle.
Tolerances: the network's own 1e-5 (values) and 1e-4 (gradient)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,hidden,n_out,batch", [(1, 1, 1, 1), (384, 256, 16, 127), (384, 256, 16, 128),
                                                     (120, 64, 4, 129), (121, 65, 5, 33), (208, 72, 8, 255),
                                                     (384, 256, 16, 2049), (130, 129, 3, 1500)])
def test_network_products_at_tile_edges(dcmod, cuda_ok, n_in, hidden, n_out, batch):
    import torch
    from oracle import mlp as M
    rng = np.random.default_rng(n_in + hidden + batch)
    n = dcmod.mlp_param_count(n_in, hidden, n_out)
    p = (rng.standard_normal(n) * 0.1).astype(np.float32)
    x = rng.uniform(-1, 1, (batch, n_in)).astype(np.float32)
    t = rng.standard_normal((batch, n_out)).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    work = torch.empty(dcmod.mlp_workspace_floats(n_in, hidden, n_out, batch), dtype=torch.float32, device="cuda")
    y = torch.empty((batch, n_out), dtype=torch.float32, device="cuda")
    dcmod.mlp_forward(n_in, hidden, n_out, dev(p), dev(x), y, work)
    outs = []
    for _ in range(2):
        grad = torch.full((n,), float("nan"), dtype=torch.float32, device="cuda")
        loss = torch.empty(1, dtype=torch.float32, device="cuda")
        dcmod.mlp_loss_grad(n_in, hidden, n_out, dev(p), dev(x), dev(t), grad, loss, work)
        outs.append((grad.cpu().numpy(), loss.item()))
    assert np.array_equal(outs[0][0], outs[1][0]) and outs[0][1] == outs[1][1]    # a fixed order
    ry, _ = M.forward(p.astype(np.float64), x, n_in, hidden, n_out)
    rl, rg = M.loss_grad(p.astype(np.float64), x, t, n_in, hidden, n_out)
    assert np.abs(y.cpu().numpy() - ry).max() <= 1e-5 * max(1.0, np.abs(ry).max())
    assert abs(outs[0][1] - rl) <= 1e-5 * rl
    assert np.abs(outs[0][0] - rg).max() <= 1e-4 * np.abs(rg).max()
