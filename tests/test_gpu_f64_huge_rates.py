"""The FP64 form at rates far past any physical W dt: every state whose rate
is huge empties into the first one above it whose rate is not, and nothing
becomes infinite or NaN on the way."""
import numpy as np
import pytest
import torch
from scipy.linalg import expm

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species, oracle_species

pytestmark = pytest.mark.gpu

HUGE, FLAT = 1e19, 700.0  # W dt of a state that empties at once; of one that may keep something


def crossings(spo, Z):
    """Fields at which two neighbouring states' rates are equal to rounding."""
    out = []
    for k in range(Z - 1):
        E = np.logspace(1.5, 5, 4001)
        r = oracle.rates(spo, E, k, k + 2)
        d = np.where((r > 0).all(0), np.sign(r[0] - r[1]), 0)
        for i in np.flatnonzero(d[:-1] * d[1:] < 0):
            a, b = E[i], E[i + 1]
            for _ in range(60):
                m = 0.5 * (a + b)
                q = oracle.rates(spo, np.array([m]), k, k + 2)[:, 0]
                a, b = (m, b) if np.sign(q[0] - q[1]) == d[i] else (a, m)
            out += [a, b, a * (1 + 1e-9), a * (1 - 1e-12)]
    return np.array(out)


def limit(lam, v):
    """exp of the window's chain with states of lam > HUGE emptied at once."""
    w = len(v)
    keep = [r for r in range(w) if r == w - 1 or lam[r] <= HUGE]
    x = np.zeros(len(keep))
    for r in range(w):
        x[next(i for i, s in enumerate(keep) if s >= r)] += v[r]
    A = np.zeros((len(keep),) * 2)
    for i, s in enumerate(keep[:-1]):
        A[i, i] = -lam[s]
        A[i + 1, i] = lam[s]
    out = np.zeros(w)
    out[keep] = expm(A) @ x
    return out


@pytest.mark.parametrize("n", [4000, 170_000])
@pytest.mark.parametrize("dt", [1e34, 1e40, 1e150, 1e300])
def test_huge_rates_empty_their_states(dt, n):
    """Both grids of the FP64 form (one cell per lane, and the class queues).
    1e-12, the form's bar."""
    sd = W.nitrogen()
    spo = oracle_species(sd)
    rng = np.random.default_rng(5)
    E = 10.0 ** rng.uniform(0.3, 5, 1000)
    x = crossings(spo, sd.Z)
    assert len(x) >= 8
    E = np.concatenate([E, np.repeat(x, 10)])
    m = len(E)
    lo = rng.integers(0, 3, m)
    hi = np.minimum(lo + rng.integers(1, 6, m), sd.Z)
    N = np.zeros((sd.Z + 1, m))
    for c in range(m):
        N[lo[c]:hi[c] + 1, c] = rng.dirichlet(np.ones(hi[c] - lo[c] + 1))
    R = oracle.rates(spo, E, 0, sd.Z) * dt
    assert (R > 4e38).mean() > 0.1 or dt < 1e40
    at = np.arange(n) % m
    Nd = torch.tensor(np.ascontiguousarray(N[:, at]), device="cuda")
    l = torch.tensor(lo[at].astype(np.uint8), device="cuda")
    h = torch.tensor(hi[at].astype(np.uint8), device="cuda")
    dne = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    ionize.step(gpu_species(sd), torch.tensor(E[at], device="cuda"), Nd, l, h, dt, dne,
                flags=ionize.ION_F64_PLAIN | ionize.ION_NO_WINDOW_UPDATE)
    out, dne = Nd.cpu().numpy(), dne.cpu().numpy()  # (planes, cells)
    assert np.isfinite(out).all() and np.isfinite(dne).all()
    assert np.array_equal(out[:, :m], out[:, at][:, :m])
    seen = 0
    for c in range(min(n, m)):
        lam = R[lo[c]:hi[c], c]
        if np.any((lam > FLAT) & (lam <= HUGE)):
            continue  # neither empty at once nor a chain the reference takes
        v = N[lo[c]:hi[c] + 1, c]
        ref = limit(lam, v)
        assert np.abs(out[lo[c]:hi[c] + 1, c] - ref).max() <= 1e-12
        assert abs(dne[c] - np.arange(len(v)) @ (ref - v)) <= 1e-12 * len(v)
        seen += 1
    assert seen > m // 2
