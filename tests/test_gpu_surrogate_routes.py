"""ion_step_surrogate's two routes: the streaming kernel that leaves the cells
the network may serve to a list (arrays it takes, a surrogate with validation
bounds, the paper's window rule), and the network kernel over all cells (any
other call).  Both against the oracle, and against each other."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, surrogate as S, workloads as W
from test_gpu_step import check, gpu_species, oracle_species

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def short_net():
    sd = W.argon_like()
    sp = gpu_species(sd)
    return sd, sp, S.build(sp, steps=1500, seed=31)[0]


def shifted(t, skip):
    """The values of t behind `skip` elements of another buffer."""
    b = torch.empty(t.numel() + skip, dtype=t.dtype, device="cuda")[skip:].view(t.shape)
    return b.copy_(t)


def step(net, wl, E, lo, hi, G, skip=0, pop_tol=1e-6, window=None):
    n = wl.ncells
    N, E = wl.N.cuda(), E.cuda()
    l, h = shifted(lo.cuda(), skip), shifted(hi.cuda(), skip)
    dne = torch.full((n,), 7.0, device="cuda")
    ws = net.step(E, N, l, h, 0.05, dne, n_gas=G, pop_tol=pop_tol, window=window)
    torch.cuda.synchronize()
    out = dict(N=N.double().cpu().numpy(), lo=l.cpu().numpy(), hi=h.cpu().numpy(),
               dne=dne.double().cpu().numpy())
    return out, ionize.surrogate_counters(ws), ionize.counters(ws)[1]


@pytest.mark.parametrize("n", [1, 63, 64, 65, 129, 4099, 150_001])
def test_routes_agree_with_the_oracle(short_net, n):
    """Aligned arrays (the list) and windows one byte off (all cells): each
    within the FP32 bar of the oracle, the same counts of cells, and as many
    on the network up to one in a thousand (the routes evaluate Eq. 1 in two FP32
    forms, which can only matter to a cell the network would have to be
    further off than twice its bound to serve)."""
    sd, sp, net = short_net
    wl = W.ladder_cells(sd, n, 41, block=64)
    E = wl.E.clone()
    E[::11] *= 1e-2  # below the window's rates
    E[1::97] = 0.0
    E[2::97] = 3.0     # outside the trained range
    E[3::97] = 2.0e5
    E[5::97] = -E[5::97]
    G = torch.full((n,), 1.0, device="cuda")
    No, loo, hio, dneo = oracle.step(oracle_species(sd), E.double().numpy(),
                                     wl.N[:, :n].double().numpy(), 0.05, wl.lo.numpy(),
                                     wl.hi.numpy())
    ref = dict(N=No, lo=loo, hi=hio, dne=dneo)
    counts = []
    for skip in (0, 1):
        out, (n_net, n_plain, timeout), bad = step(net, wl, E, wl.lo, wl.hi, G, skip)
        check(out, ref, wl.lo, wl.hi, ionize.ION_F32, n=n, sd=sd, E=E.double().numpy())
        assert timeout == 0 and bad == 0
        assert n_net + n_plain == int((wl.hi > wl.lo).sum())
        counts.append(n_net)
    assert abs(counts[0] - counts[1]) <= max(1, n // 1000)
    if n > 4000:
        assert counts[0] > n // 20  # the network is used


def test_routes_on_odd_windows(short_net):
    """Single states, invalid windows and a gas density, on both routes: the
    invalid cells are counted and left alone, dne scales."""
    sd, sp, net = short_net
    n = 20_011
    wl = W.ladder_cells(sd, n, 43, block=64)
    lo, hi = wl.lo.clone(), wl.hi.clone()
    lo[::101], hi[::101] = 4, 4
    lo[7::101], hi[7::101] = 9, 3
    lo[9::101], hi[9::101] = 15, 19
    valid = (lo <= hi) & (hi <= sd.Z) & (hi.int() - lo.int() < 6)
    G = 0.5 + torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    one = torch.ones(n, device="cuda")
    res = [step(net, wl, wl.E, lo, hi, g, skip) for g, skip in ((G, 0), (G, 1), (one, 0))]
    (a, ca, bad_a), (b, cb, bad_b), (c, _, _) = res
    assert bad_a == bad_b == int((~valid).sum())
    assert ca[0] + ca[1] == cb[0] + cb[1] == int((valid & (hi > lo)).sum())
    inv = ~valid.numpy()
    for o in (a, b):
        assert np.array_equal(o["N"][:, :n][:, inv], wl.N[:, :n].double().numpy()[:, inv])
        assert np.all(o["dne"][inv] == 7.0)
    # two results within the FP32 bar of the same exact ones
    assert np.abs(a["N"] - b["N"]).max() <= 4e-6
    g = G.double().cpu().numpy()
    ok = valid.numpy()
    assert np.allclose(a["dne"][ok], (c["dne"] * g)[ok], rtol=1e-6, atol=0)


@pytest.mark.parametrize("pop_tol,window", [(0.0, None), (1e30, None),
                                            (1e-6, {"w_min": 2, "w_max": 6, "eps_grow": 1e-6})])
def test_routes_at_the_ends(short_net, pop_tol, window):
    """pop_tol 0 never uses the network; a huge one uses it wherever the
    field is in range and no rate is stiff; the adaptive rule takes the
    network kernel over all cells whatever the alignment: equal bits."""
    sd, sp, net = short_net
    n = 30_000
    wl = W.ladder_cells(sd, n, 44, block=64)
    a, ca, _ = step(net, wl, wl.E, wl.lo, wl.hi, None, 0, pop_tol, window)
    b, cb, _ = step(net, wl, wl.E, wl.lo, wl.hi, None, 1, pop_tol, window)
    assert ca[0] + ca[1] == cb[0] + cb[1] == n
    if pop_tol == 0.0:
        assert ca[0] == cb[0] == 0
    elif window is None:
        assert ca == cb and ca[0] > n // 2
    if window is not None or pop_tol > 1:
        # the same cells, kernels and records in both
        for k in ("N", "lo", "hi", "dne"):
            assert np.array_equal(a[k], b[k])
