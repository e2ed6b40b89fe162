"""The training step at batches around its row pairs and its staging chunk of
256 rows, and inputs that are only 4-byte aligned; reference and tolerance are
those of the network's other tests."""

import numpy as np
import pytest

from paper_2401_02756_gb300 import dbg
from test_gpu_mlp import (GAMMA, _lib, case, dev, magnitudes, mlp, pytestmark,  # noqa: F401
                          work)


@pytest.mark.parametrize("batch", [1, 2, 255, 256, 257, 513])
def test_train_step_gradients_at_batch_edges(batch):
    import torch
    p, x, t = case(200 + batch, batch)
    G = torch.zeros(mlp.N_PARAMS, device="cuda")
    M, V = torch.zeros_like(G), torch.zeros_like(G)
    dbg.mlp_train_step(dev(p), G, M, V, 1, 1e-3, dev(x), dev(t), work(batch))
    _, ref = mlp.loss_and_grads(p, x, t)
    g = G.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= GAMMA * magnitudes(p, x, t)[3])
    assert np.array_equal(g == 0.0, ref == 0.0)  # the same ReLU branches and dead inputs
    one_m_b1 = float(np.float32(1) - np.float32(0.9))
    assert np.allclose(M.cpu().numpy(), one_m_b1 * g, rtol=1e-6, atol=0)


def test_unaligned_rows_give_the_same_output():
    import torch
    p, x, _ = case(900, 5)
    outs = []
    for shift in (0, 1, 3):
        X = torch.zeros(5 * mlp.IN + shift, device="cuda")[shift:]
        P = torch.zeros(dbg.MLP_PARAMS + shift, device="cuda")[shift:]
        X.copy_(dev(x).view(-1))
        P.copy_(dev(p))
        y = torch.empty(5, device="cuda")
        dbg.mlp_forward(P, X, y, work(5))
        outs.append(y.cpu())
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
