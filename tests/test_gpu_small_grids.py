"""Small FP32 grids run one cell per lane in a single kernel; a launch shape
asks for the streaming kernels.  Both on the same cells: each within the FP32
bar of the oracle, with the same cells counted as invalid, stiff and done
with FP64 coefficients."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species, oracle_species, window_ties

pytestmark = pytest.mark.gpu

ADAPT = {"w_min": 2, "w_max": 6, "eps_grow": 1e-6}


def words(ws):
    return ws[:44].cpu().view(torch.int32).tolist()


@pytest.mark.parametrize("name", ["N", "Kr-like"])
@pytest.mark.parametrize("flags,window", [(0, None), (0, ADAPT), (ionize.ION_NO_WINDOW_UPDATE, None),
                                          (ionize.ION_CONSERVATION_CHECK, None),
                                          (ionize.ION_NO_FP64_FALLBACK, None),
                                          (ionize.ION_FORCE_FP64_COEF, None)])
@pytest.mark.parametrize("n", [1, 31, 64, 19_968, 20_011])
def test_direct_and_streaming_grids(name, flags, window, n):
    sd = W.nitrogen() if name == "N" else W.krypton_like()
    sp = gpu_species(sd)
    wl = W.ladder_cells(sd, n, 17, block=64)
    lo, hi = wl.lo.clone(), wl.hi.clone()
    lo[5::211], hi[5::211] = 2, 2
    lo[7::211], hi[7::211] = 6, 1
    lo[9::211], hi[9::211] = sd.Z - 1, sd.Z + 1
    E = wl.E.clone()
    E[11::211] = 0.0
    E[13::211] *= -1.0
    ld = n + 3  # rows that are not 16-byte aligned
    N0 = torch.zeros((sd.Z + 1, ld))
    N0[:, :n] = wl.N[:, :n]
    G = 0.5 + torch.rand(n, generator=torch.Generator().manual_seed(3))
    valid = ((lo <= hi) & (hi <= sd.Z)).numpy()
    kw = {} if window is None else dict(policy=oracle.WINDOW_ADAPTIVE, w_min=2, w_max=6,
                                        eps_grow=1e-6)
    ref = oracle.step(oracle_species(sd), E.double().numpy()[valid],
                      N0[:, :n].double().numpy()[:, valid], 0.05, lo.numpy()[valid],
                      hi.numpy()[valid], window_update=not flags & ionize.ION_NO_WINDOW_UPDATE, **kw)
    seen = []
    for shape in (None, (2, 8, 0), (1, 4, 0)):
        Nd, l, h = N0.cuda(), lo.cuda(), hi.cuda()
        dne = torch.full((n,), 7.0, device="cuda")
        ws = ionize.step_batched([(sp, E.cuda(), Nd, l, h, dne, G.cuda())], 0.05, flags=flags,
                                 shape=shape, window=window)
        torch.cuda.synchronize()
        out = Nd.double().cpu().numpy()
        err = np.abs(out[:, :n][:, valid] - ref[0])
        assert err.max() <= 2e-6, err.max()
        w = (hi.int() - lo.int() + 1).numpy()[valid]
        g = G.double().numpy()[valid]
        d = dne.double().cpu().numpy()
        assert np.all(np.abs(d[valid] / g - ref[3]) <= np.maximum(w - 1, 1) * 2e-6)
        # nothing but the valid cells' windows is written
        assert np.array_equal(out[:, :n][:, ~valid], N0[:, :n].double().numpy()[:, ~valid])
        assert np.all(d[~valid] == 7.0) and np.all(out[:, n:] == 0)
        # the rule on the GPU's own populations, bit for bit; windows other than
        # the oracle's only where a population straddles a threshold
        # (a single state keeps its window here; the oracle's adaptive rule lets it grow)
        if not flags & ionize.ION_NO_WINDOW_UPDATE:
            m = valid & (hi > lo).numpy()
            r = m[valid]
            window_ties(sd, E.double().numpy()[m], out[:, :n][:, m], ref[0][:, r],
                        lo.numpy()[m], hi.numpy()[m], l.cpu().numpy()[m],
                        h.cpu().numpy()[m], ref[1][r], ref[2][r], 1e-6, True, policy=window)
            assert torch.equal(l.cpu()[hi == lo], lo[hi == lo])
            assert torch.equal(h.cpu()[hi == lo], hi[hi == lo])
        else:
            assert torch.equal(l.cpu(), lo) and torch.equal(h.cpu(), hi)
        h_ = words(ws)
        assert h_[1] == int((~valid).sum())
        seen.append((h_[0], h_[2]))
        if flags & ionize.ION_CONSERVATION_CHECK:
            change = np.abs(out[:, :n].sum(0) - N0[:, :n].double().numpy().sum(0)).max()
            assert abs(ionize.conservation_change(ws) - change) <= 1e-9
    # the counts of cells with FP64 coefficients agree with the streaming
    # kernels', and of stiff cells where no partial chunk adds records
    assert seen[0][0] == seen[1][0] or flags & ionize.ION_FORCE_FP64_COEF
    if n % 64 == 0:
        assert seen[0] == seen[1]


def test_small_batch_of_species():
    """Three species in one small call: the jobs' cells lie one after
    another in the grid, with a block shared by two jobs."""
    jobs_a, jobs_b = [], []
    for sd, n in ((W.nitrogen(), 1000), (W.argon_like(), 37), (W.krypton_like(), 5003)):
        sp = gpu_species(sd)
        wl = W.ladder_cells(sd, n, 19, block=64, device="cuda")
        for jobs in (jobs_a, jobs_b):
            jobs.append((sp, wl.E, wl.N.clone(), wl.lo.clone(), wl.hi.clone(),
                         torch.empty(n, device="cuda")))
    ionize.step_batched(jobs_a, 0.05)
    for j in jobs_b:
        ionize.step(*j[:5], 0.05, j[5])
    for a, b in zip(jobs_a, jobs_b):
        for x, y in zip(a[2:], b[2:]):
            # the widest window of a warp bounds the loops, not the result
            assert torch.equal(x, y)
