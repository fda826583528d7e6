"""Short queues of the FP64-coefficient pass."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species, oracle_species

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stiff", [1, 3, 1217, 5003])
def test_short_fp64_queues(stiff):
    """Queues of fewer entries than the grid has warps, and of a few per warp: every
    queued cell is done once, within the FP32 bar of the oracle."""
    sd = W.argon_like()
    n = 410_000  # past the small grids, which queue nothing
    wl = W.ladder_cells(sd, n, 5, device="cpu")
    Wr = oracle.rates(oracle_species(sd), wl.E.double().numpy(), 0, sd.Z) * 0.05
    lo, hi = wl.lo.numpy().astype(int), wl.hi.numpy().astype(int)
    k = np.arange(sd.Z)[:, None]
    lmax = np.where((k >= lo) & (k < hi), Wr, 0.0).max(0)
    cells = np.flatnonzero(lmax > 1.1)[:stiff]
    assert len(cells) == stiff
    E = torch.zeros(n)
    E[cells] = wl.E[cells]
    N = wl.N.cuda()
    l, h = wl.lo.cuda(), wl.hi.cuda()
    dne = torch.empty(n, device="cuda")
    ws = ionize.step(gpu_species(sd), E.cuda(), N, l, h, 0.05, dne,
                     flags=ionize.ION_FORCE_FP64_COEF | ionize.ION_NO_WINDOW_UPDATE)
    assert ionize.counters(ws) == (stiff, 0)
    No, _, _, do = oracle.step(oracle_species(sd), E[cells].double().numpy(),
                               wl.N[:, cells].double().numpy(), 0.05, wl.lo.numpy()[cells],
                               wl.hi.numpy()[cells], window_update=False)
    assert np.abs(N.cpu()[:, cells].double().numpy() - No).max() <= 2e-6
    rest = np.setdiff1d(np.arange(n), cells)
    assert torch.equal(N.cpu()[:, rest], wl.N[:, rest])
