"""Gradient and predictions of the smoothing-length network at the edges of its
tiles: one sample, around one tile of 64 and of 16, and more tiles than a
persistent grid of two blocks per SM holds at once.  Against the FP64 oracle on
the BF16 operands, with the tolerance of the other network tests (three times it
below a tile, where the errors of single samples do not average)."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl

from test_gpu_mlp import BF16_RTOL, _bf16, _data, _weights_as_used

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 17, 63, 64, 65, 2 * 152 * 64 - 1, 2 * 152 * 64 + 65, 45000])
def test_gradient_and_predictions_at_tile_edges(n):
    import torch
    X, y = _data(n, 50 + n % 13)
    y = (y + 3.0).astype(np.float32)   # no sample is predicted exactly
    M = nl.MLP(seed=7)
    Pu = _weights_as_used(M.get_params())
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    wd = torch.ones(n, dtype=torch.float32, device="cuda")
    pred = torch.full((n + 8,), -77.0, dtype=torch.float32, device="cuda")
    M.predict(Xd, pred[:n])
    want = orc.mlp_forward(_bf16(X).astype(np.float64), Pu)
    got = pred.cpu().numpy()
    assert np.max(np.abs(got[:n] - want)) <= BF16_RTOL * (np.abs(want).max() + 1.0)
    assert np.all(got[n:] == -77.0)
    g = torch.empty(M.nparams(), dtype=torch.float32, device="cuda")
    loss = M.grad(Xd, yd, wd, g)
    lw, gw = orc.mlp_loss_grad(_bf16(X).astype(np.float64), y.astype(np.float64), Pu)
    tol = BF16_RTOL * (3.0 if n < 64 else 1.0)
    assert abs(loss - lw) <= tol * lw
    assert np.linalg.norm(g.cpu().numpy() - gw) <= tol * np.linalg.norm(gw)
    M.free()
