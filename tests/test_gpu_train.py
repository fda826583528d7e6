"""The training kernel at the edges of its tiles: one sample, tiles of 64
samples that are full, short or spread over several per block, and output
counts around each padded width, against the FP64 reference network."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2202_10647_gb300 import ionize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 16, 17, 48, 63])
@pytest.mark.parametrize("B", [1, 63, 64, 65, 9729, 30001])
def test_loss_grad_tiles(K, B):
    """FP32 sums of B samples: 2e-5 of the largest gradient component, the
    tolerance of the other sizes' test."""
    rng = np.random.default_rng(100 * K + B % 97)
    P = rng.normal(0.0, 0.5, omlp.nparams(K)).astype(np.float32)
    x = rng.uniform(-1, 1, B).astype(np.float32)
    t = rng.normal(0, 1, (B, K)).astype(np.float32)
    L, g = omlp.loss_grad(P.astype(np.float64), K, x.astype(np.float64), t.astype(np.float64))
    Pd, xd, td = (torch.tensor(a, device="cuda") for a in (P, x, t))
    # a workspace of exactly the asked size, and a parameter array that is
    # only 4-byte aligned
    ws = ionize.mlp_workspace(K, B)
    ws.fill_(0xFF)  # NaN: nothing unwritten is summed
    Po = torch.empty(P.size + 1, device="cuda")[1:]
    Po.copy_(Pd)
    loss, grad = ionize.mlp_loss_grad(Po, K, xd, td, ws=ws)
    assert abs(float(loss) - L) <= 2e-5 * L
    assert np.abs(grad.double().cpu().numpy() - g).max() <= 2e-5 * np.abs(g).max()
    loss2, grad2 = ionize.mlp_loss_grad(Pd, K, xd, td)
    assert torch.equal(grad, grad2) and torch.equal(loss, loss2)
