"""A cell's result does not depend on the size of the call: small grids (one
cell per lane, a single kernel) give the streaming kernels' bits, so that a
caller may step a grid in ranges of whole 64-cell chunks."""
import pytest
import torch

from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species

pytestmark = pytest.mark.gpu

GASES = {"N": W.nitrogen, "Ar-like": W.argon_like, "Kr-like": W.krypton_like}
ADAPT = {"w_min": 2, "w_max": 6, "eps_grow": 1e-6}


def cells(sd, n, seed):
    """Ladder cells with cold runs, single states, invalid windows, zero and
    negative fields, populations at the thresholds, and a gas density."""
    wl = W.ladder_cells(sd, n, seed, block=64, device="cuda")
    E, lo, hi = wl.E.clone(), wl.lo.clone(), wl.hi.clone()
    i = torch.arange(n, device="cuda")
    E[(i // 64) % 5 == 2] *= 1e-3  # cold chunks
    E[(i // 32) % 7 == 3] *= 0.3   # cold halves beside warm ones
    E[11::211] = 0.0
    E[13::211] *= -1.0
    lo[5::211], hi[5::211] = 2, 2
    lo[7::211], hi[7::211] = 6, 1
    lo[9::211], hi[9::211] = sd.Z - 1, sd.Z + 1
    ok = i[17::211]  # a lowest state at the threshold
    wl.N[lo[ok].long(), ok] = 1e-6 * (0.5 + torch.rand(
        len(ok), device="cuda", generator=torch.Generator("cuda").manual_seed(seed)))
    G = 0.5 + torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    return wl.N[:, :n], E, lo, hi, G


def run(sp, N, E, lo, hi, G, ld, **kw):
    n = E.numel()
    Nd = torch.zeros((N.shape[0], ld), device="cuda")
    Nd[:, :n] = N
    l, h = lo.clone(), hi.clone()
    dne = torch.full((n,), 7.0, device="cuda")
    ws = ionize.step_batched([(sp, E, Nd, l, h, dne, G)], 0.05, **kw)
    return (Nd, l, h, dne), ws[:44].cpu().view(torch.int32).tolist()


@pytest.mark.parametrize("name", sorted(GASES))
@pytest.mark.parametrize("flags,window", [(0, None), (0, ADAPT), (ionize.ION_NO_WINDOW_UPDATE, None),
                                          (ionize.ION_CONSERVATION_CHECK, None),
                                          (ionize.ION_CONSERVATION_CHECK, ADAPT),
                                          (ionize.ION_NO_FP64_FALLBACK, None),
                                          (ionize.ION_FORCE_FP64_COEF, None)])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 20_011, 399_936])
def test_small_grids_give_the_streaming_bits(name, flags, window, n):
    """Against the lean kernel (rows of a multiple of four cells) and the
    general one (odd rows)."""
    sd = GASES[name]()
    sp = gpu_species(sd)
    args = cells(sd, n, 23)
    a, ha = run(sp, *args, ld=n, flags=flags, window=window)
    for ld in ((n + 3) // 4 * 4, n + 1 + n % 2):
        b, hb = run(sp, *args, ld=ld, flags=flags, window=window, shape=(2, 8, 0))
        assert torch.equal(a[0], b[0][:, :n])
        for x, y in zip(a[1:], b[1:]):
            assert torch.equal(x, y)
        assert (ha[0], ha[1], ha[10]) == (hb[0], hb[1], hb[10])
        assert ha[2] == hb[2] or n % 64  # a partial chunk's cells are records there


@pytest.mark.parametrize("name", sorted(GASES))
def test_ranges_give_the_whole_call(name):
    sd = GASES[name]()
    sp = gpu_species(sd)
    n = 500_027
    N, E, lo, hi, G = cells(sd, n, 24)
    a, _ = run(sp, N, E, lo, hi, G, ld=n + 1)
    Nd = torch.zeros((sd.Z + 1, n + 1), device="cuda")
    Nd[:, :n] = N
    l, h, dne = lo.clone(), hi.clone(), torch.full((n,), 7.0, device="cuda")
    for c0 in range(0, n, 100_032):
        ionize.step(sp, E, Nd, l, h, 0.05, dne, n_gas=G, offset=c0, ncells=min(100_032, n - c0))
    for x, y in zip(a, (Nd, l, h, dne)):
        assert torch.equal(x, y)


def test_small_batches_give_the_streaming_bits():
    """Jobs of several species, with partial last chunks and an empty one."""
    out = []
    for shape in (None, (2, 8, 0)):
        jobs = []
        for name, n in (("N", 1000), ("Ar-like", 0), ("Ar-like", 37), ("Kr-like", 5003), ("N", 64)):
            sd = GASES[name]()
            N, E, lo, hi, G = cells(sd, max(n, 1), 25)
            jobs.append((gpu_species(sd), E[:n], N[:, :max(n, 1)].clone(), lo[:n].clone(),
                         hi[:n].clone(), torch.full((n,), 7.0, device="cuda"), G[:n]))
        ionize.step_batched(jobs, 0.05, shape=shape)
        out.append(jobs)
    for a, b in zip(*out):
        for x, y in zip(a[2:6], b[2:6]):
            assert torch.equal(x, y)
