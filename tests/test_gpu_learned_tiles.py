"""The training gradient at the edges of its 128-sample tiles, and over several tiles.

Tolerance: as in the gradient test over whole batches, the BF16 rounding (unit roundoff 2^-9) of
the weights, the layer inputs and the backward operands, 4e-2 normwise per parameter block; the
loss is held to 1e-2. Slots past the batch must contribute nothing: the same samples, drawn once
more behind a longer array of pairs filled with NaN, give the same bits.
"""
import numpy as np
import pytest

import oracle.mlp as M
from _gpu_common import host, rel, require_gpu
from test_gpu_learned import f32, theta_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 17, 127, 128, 129, 1153])
def test_gradient_at_tile_edges(batch):
    torch, P = require_gpu()
    th = theta_np(5)
    rng = np.random.default_rng(6)
    X = rng.standard_normal((batch, M.N_IN)) / np.sqrt(M.N_IN)
    T = rng.standard_normal((batch, M.N_OUT)) * 0.5
    th32, X32, T32 = (a.astype(np.float32).astype(np.float64) for a in (th, X, T))
    loss_o, g_o = M.loss_and_grad(th32, X32, T32)
    out = []
    for pad in (0, 200):
        grad = torch.empty(M.n_params(), dtype=torch.float32, device="cuda")
        loss = torch.zeros(1, dtype=torch.float32, device="cuda")
        Xp = np.concatenate([X, np.full((pad, M.N_IN), np.nan)])
        Tp = np.concatenate([T, np.full((pad, M.N_OUT), np.nan)])
        P.dg_mlp_grad(f32(th), f32(Xp), f32(Tp), batch, grad, loss)
        out.append((host(grad).astype(np.float64), float(host(loss)[0])))
    (g, loss), (g2, loss2) = out
    assert np.array_equal(g, g2) and loss == loss2
    assert abs(loss - loss_o) / loss_o < 1e-2
    go, gg = M.unpack(g_o), M.unpack(g)
    for name, _ in M.SHAPES:
        assert rel(gg[name], go[name]) < 4e-2, name
