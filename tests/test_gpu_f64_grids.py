"""The FP64 form's two grids: a call large enough for the class queues against
the same cells stepped in ranges that run one cell per lane.  A cell's
arithmetic is the same in both, so every output is equal bit for bit."""
import pytest
import torch

from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [None, {"w_min": 2, "w_max": 6, "eps_grow": 1e-6}])
@pytest.mark.parametrize("flags", [0, ionize.ION_NO_WINDOW_UPDATE, ionize.ION_CONSERVATION_CHECK])
def test_queued_and_direct_grids_agree(window, flags):
    n = 420_011
    sd = W.krypton_like()
    sp = gpu_species(sd)
    wl = W.ladder_cells(sd, n, 9, device="cuda")
    lo, hi = wl.lo.clone(), wl.hi.clone()
    lo[::1009], hi[::1009] = 3, 3    # a single state
    lo[5::2003], hi[5::2003] = 9, 4  # no window
    lo[7::4001], hi[7::4001] = 30, 37  # past the top
    E = wl.E.double()
    E[11::3001] = 0.0
    E[13::3001] = float("inf")
    E[17::3001] = -E[17::3001]
    G = 0.5 + torch.rand(n, device="cuda", dtype=torch.float64,
                         generator=torch.Generator(device="cuda").manual_seed(1))
    f = flags | ionize.ION_F64_PLAIN

    def state():
        return wl.N.double(), lo.clone(), hi.clone(), torch.full((n,), 7.0, device="cuda",
                                                                 dtype=torch.float64)

    a, b = state(), state()
    ws = ionize.step(sp, E, a[0], a[1], a[2], 0.05, a[3], n_gas=G, flags=f, window=window)
    bad = ionize.counters(ws)[1]
    change = ionize.conservation_change(ws)
    part_bad, part_change = 0, 0.0
    for c0 in range(0, n, 100_003):
        m = min(100_003, n - c0)
        w = ionize.step(sp, E, b[0], b[1], b[2], 0.05, b[3], n_gas=G, flags=f, window=window,
                        offset=c0, ncells=m)
        part_bad += ionize.counters(w)[1]
        part_change = max(part_change, ionize.conservation_change(w))
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert bad == part_bad == int(((lo > hi) | (hi > sd.Z)).sum())
    if flags & ionize.ION_CONSERVATION_CHECK:
        assert change == part_change
