"""The surrogate's training data at the edges of its kernels' tiles and of
their arithmetic: ion_log2_rates against the oracle, ion_mlp_inputs and
ion_mlp_standardize against numpy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize
from paper_2202_10647_gb300 import surrogate as S
from paper_2202_10647_gb300 import workloads as W
from test_gpu_step import gpu_species, oracle_species

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k_lo,k_hi,pad", [(1, 0, 36, 0), (255, 3, 4, 0), (256, 0, 36, 1),
                                             (257, 17, 36, 5), (1023, 35, 36, 0)])
def test_log2_rates_tile_edges(n, k_lo, k_hi, pad):
    """Blocks of 256 cells, threads in multiples of the state count, rows
    with a stride: within 1e-10 of the oracle in log2 (1e-12 relative in W),
    the floor exactly, nothing written outside."""
    sd = W.krypton_like()
    sp = gpu_species(sd)
    rng = np.random.default_rng(n)
    E = (10.0 ** rng.uniform(-7, 6, n)).astype(np.float32)
    E[:: 7] = 0.0
    K, floor = k_hi - k_lo, -60.0
    buf = torch.full((n, K + pad), 7.0, dtype=torch.float64, device="cuda")
    rc = ionize.lib().ion_log2_rates(sp.handle, torch.tensor(E, device="cuda").data_ptr(), n,
                                     k_lo, k_hi, floor, buf.data_ptr(), K + pad, None)
    assert rc == 0
    torch.cuda.synchronize()
    y = buf.cpu().numpy()
    with np.errstate(divide="ignore"):
        ref = np.maximum(np.log2(oracle.rates(oracle_species(sd), E.astype(np.float64), 0, sd.Z)),
                         floor).T[:, k_lo:k_hi]
    assert np.abs(y[:, :K] - ref).max() <= 1e-10
    assert np.all(y[:, :K][ref == floor] == floor)
    assert np.all(y[:, K:] == 7.0)


def test_mlp_inputs_special_fields():
    """Zero, denormal, infinite and NaN fields, and both ends of the range,
    as numpy's log2 gives them (NaN: -1)."""
    E = np.array([0.0, -0.0, 1e-45, -1.1754942e-38, 1.1754944e-38, 3.4028235e38, np.inf, -np.inf,
                  np.nan, 10.0, 1e5, 9.9999, 100001.0, 1.0], dtype=np.float32)
    l2lo, l2hi = S.log2_range()
    for lo, hi in ((l2lo, l2hi), (-149.0, 128.0)):
        x = ionize.mlp_inputs(torch.tensor(E, device="cuda"), lo, hi).cpu().numpy()
        with np.errstate(divide="ignore", invalid="ignore"):
            v = 2.0 * (np.log2(np.abs(E.astype(np.float64))) - lo) / (hi - lo) - 1.0
        ref = np.where(np.isnan(v), -1.0, np.clip(v, -1.0, 1.0)).astype(np.float32)
        # float rounding of an FP64 value within a few 1e-16: one ulp where it is a tie
        assert np.all(np.abs(x - ref) <= np.spacing(np.abs(ref)))


@pytest.mark.parametrize("K", [1, 2, 18, 63])
@pytest.mark.parametrize("slices", [0.1, 1, 2.5])
def test_mlp_standardize_slices(K, slices):
    """Row counts around the slices the moments are summed by (0.1: the
    one-block-per-column form), and columns outside the range of the FP32
    pairs: constant, zero, huge, tiny, far from their spread.  The targets
    are the FP64 quotient's float, value for value."""
    rows = 256 // K * 32
    for n in {max(2, int(rows * slices) - 1), max(2, int(rows * slices)), int(rows * slices) + 3}:
        rng = np.random.default_rng(n * 64 + K)
        Y = rng.normal(0.0, 1.0, (n, K)) * rng.uniform(0.1, 30.0, K) + rng.uniform(-60, 5, K)
        special = [np.full(n, -40.0), np.zeros(n), rng.normal(size=n) * 1e30,
                   rng.normal(size=n) * 1e-25, 1000.0 + rng.normal(size=n) * 1e-3,
                   np.where(np.arange(n) % 3 == 0, -40.0, rng.uniform(-40, 5, n))]
        for k, col in enumerate(special[: K - 1] if K > 1 else special[5:]):
            Y[:, k] = col
        mean, scale, T = ionize.mlp_standardize(torch.tensor(Y, device="cuda"), 1e-3)
        m, s = mean.cpu().numpy(), scale.cpu().numpy()
        # a sum of n rounds each addition by 2^-53 of at most n max|Y|
        tol = 1e-13 * np.abs(Y).max(0)
        assert np.all(np.abs(m - Y.mean(0)) <= tol)
        ref = np.maximum(Y.std(0, ddof=1), 1e-3)
        assert np.all(np.abs(s - ref) <= 1e-12 * ref + tol)
        assert np.array_equal(T.cpu().numpy(), ((Y - m) / s).astype(np.float32))
