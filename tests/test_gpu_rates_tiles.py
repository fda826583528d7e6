"""ion_rates in FP32 around its blocks of 1,024 cells, with zero, infinite and
NaN fields among them, state ranges, and a species whose rates need the
clamp and the cutoff test."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species, oracle_species

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("name", ["N", "Kr-like", "shallow"])
def test_rates_f32_blocks(n, name):
    """Within 2e-6 relative of the oracle (the FP32 rate's bar) where W dt is
    above 1e-30; for the shallow species, whose |E| power is up to 70, the
    product b log2 |E| alone rounds by 70 x 2^-24 in log2: 2e-5."""
    sd = {"N": W.nitrogen, "Kr-like": W.krypton_like}.get(
        name, lambda: W.SpeciesData("shallow", [1.0 + 0.1 * k for k in range(10)], [0] * 10,
                                    [0] * 10))()
    tol = 2e-5 if name == "shallow" else 2e-6
    sp = gpu_species(sd)
    rng = np.random.default_rng(n)
    E = (10.0 ** rng.uniform(-8, 7, n)).astype(np.float32)
    E[3::11] = 0.0
    E[5::13] *= -1.0
    E[7::101] = np.inf
    k_lo, k_hi = (0, sd.Z) if n % 2 else (sd.Z // 3, sd.Z - 1)
    W_ = torch.full((k_hi - k_lo, n + 3), 7.0, device="cuda")
    rc = ionize.lib().ion_rates(sp.handle, torch.tensor(E, device="cuda").data_ptr(), n, k_lo,
                                k_hi, W_.data_ptr(), n + 3, ionize.ION_DTYPE_F32, None)
    assert rc == 0
    torch.cuda.synchronize()
    got = W_.double().cpu().numpy()
    assert np.all(got[:, n:] == 7.0)
    got = got[:, :n]
    Eo = np.where(np.isfinite(E), np.abs(E), 0.0).astype(np.float64)  # W = 0 at infinity too
    ref = oracle.rates(oracle_species(sd), Eo, 0, sd.Z)[k_lo:k_hi]
    big = (ref * 0.05 > 1e-30) & (ref < 2.0 ** 98)
    assert np.all(np.abs(got[big] - ref[big]) <= tol * ref[big])
    assert np.all(got[ref * 0.05 <= 1e-30] * 0.05 <= 2e-30)
    assert np.all((got[ref >= 2.0 ** 98] >= 2.0 ** 97.9) & (got[ref >= 2.0 ** 98] <= 2.0 ** 99))
    assert np.all(got[:, Eo == 0] == 0)
