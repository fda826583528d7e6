"""ion_step_surrogate above the size from which the streaming kernel steps the
cells the network could not serve and lists the others: the list against the
network kernel over all cells (windows one byte off) and the oracle; smaller
calls take the latter alone."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import check, gpu_species, oracle_species
from test_gpu_surrogate_routes import short_net, step, test_routes_agree_with_the_oracle as agree

pytestmark = pytest.mark.gpu

LINE = 320_000


def listed(net, wl, n):
    """Cells left to a list by a step of the first n cells."""
    N = wl.N[:, :n].contiguous()
    lo, hi, dne = wl.lo[:n].clone(), wl.hi[:n].clone(), torch.empty(n, device="cuda")
    ws = net.step(wl.E[:n].contiguous(), N, lo, hi, 0.05, dne)
    return int(ws[36:40].cpu().view(torch.int32)[0])  # header word 9


def test_small_calls_take_one_network_kernel(short_net):
    """The two stages cost a small call more than they save: no list up to
    the line, and one from there on."""
    sd, sp, net = short_net
    wl = W.ladder_cells(sd, LINE + 64, 45, block=64, device="cuda")
    for n in (1000, 20_000, LINE):
        assert listed(net, wl, n) == 0
    assert listed(net, wl, LINE + 64) > LINE // 100


@pytest.mark.parametrize("n", [LINE, LINE + 1, LINE + 64, LINE + 127])
def test_list_agrees_with_the_oracle(short_net, n):
    agree(short_net, n)


def test_list_on_odd_windows(short_net):
    """Single states, invalid windows and a gas density: the invalid cells
    are counted and left alone, dne scales; the two routes are each within
    the FP32 bar of the same exact results."""
    sd, sp, net = short_net
    n = LINE + 11
    wl = W.ladder_cells(sd, n, 43, block=64)
    lo, hi = wl.lo.clone(), wl.hi.clone()
    lo[::101], hi[::101] = 4, 4
    lo[7::101], hi[7::101] = 9, 3
    lo[9::101], hi[9::101] = 15, 19
    valid = (lo <= hi) & (hi <= sd.Z) & (hi.int() - lo.int() < 6)
    G = 0.5 + torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    one = torch.ones(n, device="cuda")
    (a, ca, bad_a), (b, cb, bad_b), (c, _, _) = [
        step(net, wl, wl.E, lo, hi, g, skip) for g, skip in ((G, 0), (G, 1), (one, 0))]
    assert bad_a == bad_b == int((~valid).sum())
    assert ca[0] + ca[1] == cb[0] + cb[1] == int((valid & (hi > lo)).sum())
    inv = ~valid.numpy()
    for o in (a, b):
        assert np.array_equal(o["N"][:, :n][:, inv], wl.N[:, :n].double().numpy()[:, inv])
        assert np.all(o["dne"][inv] == 7.0)
    assert np.abs(a["N"] - b["N"]).max() <= 4e-6
    ok = valid.numpy()
    assert np.allclose(a["dne"][ok], (c["dne"] * G.double().cpu().numpy())[ok], rtol=1e-6, atol=0)


@pytest.mark.parametrize("pop_tol", [0.0, 1e30])
def test_list_at_the_ends(short_net, pop_tol):
    """pop_tol 0 never uses the network; a huge one uses it wherever the
    field is in range and no rate is stiff, on the same cells with equal bits."""
    sd, sp, net = short_net
    n = LINE + 640
    wl = W.ladder_cells(sd, n, 44, block=64)
    a, ca, _ = step(net, wl, wl.E, wl.lo, wl.hi, None, 0, pop_tol)
    b, cb, _ = step(net, wl, wl.E, wl.lo, wl.hi, None, 1, pop_tol)
    assert ca[0] + ca[1] == cb[0] + cb[1] == n
    if pop_tol == 0.0:
        assert ca[0] == cb[0] == 0
    else:
        assert ca == cb and ca[0] > n // 2
        for k in ("N", "lo", "hi", "dne"):
            assert np.array_equal(a[k], b[k])


def test_list_after_a_wait_that_gives_up(short_net):
    """The test hook on the list route: every cell and its dne are either
    stepped whole (those the network is not asked about) or as they were;
    the header says that the call failed, and the next calls run."""
    sd, sp, net = short_net
    n = LINE + 11
    wl = W.ladder_cells(sd, n, 47, block=64)
    E = wl.E.cuda()
    lo2, hi2, N2 = wl.lo.cuda(), wl.hi.cuda(), wl.N.cuda()
    dne2 = torch.empty(n, device="cuda")
    ionize.step(sp, E, N2, lo2, hi2, 0.05, dne2)
    net.test_timeout(True)
    try:
        for rep in range(2):
            N, lo, hi = wl.N.cuda(), wl.lo.cuda(), wl.hi.cuda()
            dne = torch.full((n,), -5.0, device="cuda")
            ws = net.step(E, N, lo, hi, 0.05, dne)
            torch.cuda.synchronize()
            n_net, n_plain, timeout = ionize.surrogate_counters(ws)
            h = ws[:44].cpu().view(torch.int32)
            kept = (dne == -5.0).cpu()
            assert timeout > 0 and n_net == 0
            assert int(kept.sum()) == int(h[9]) and n // 100 < int(h[9]) < n
            assert n_plain + int(h[9]) == n
            assert torch.equal(N.cpu()[:, :n][:, kept], wl.N[:, :n][:, kept])
            assert torch.equal(lo.cpu()[kept], wl.lo[kept])
            assert torch.equal(hi.cpu()[kept], wl.hi[kept])
            # ion_step's kernels on the others: its bits where a chunk holds no listed cell
            whole = ~kept[:n // 64 * 64].view(-1, 64).any(1).repeat_interleave(64)
            assert int(whole.sum()) > n // 10
            assert float((N - N2)[:, :n].cpu()[:, ~kept].abs().max()) <= 4e-6
            for a, b in ((N[:, :n], N2[:, :n]), (lo, lo2), (hi, hi2), (dne, dne2)):
                assert torch.equal(a[..., :len(whole)].cpu()[..., whole],
                                   b[..., :len(whole)].cpu()[..., whole])
    finally:
        net.test_timeout(False)
    N, lo, hi = wl.N.cuda(), wl.lo.cuda(), wl.hi.cuda()
    ws = net.step(E, N, lo, hi, 0.05, torch.empty(n, device="cuda"))
    torch.cuda.synchronize()
    assert ionize.surrogate_counters(ws)[2] == 0 and ionize.surrogate_counters(ws)[0] > 0
    assert float((N - N2).abs().max()) <= 4e-6
