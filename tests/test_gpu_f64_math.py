"""The fixed-point log2, reciprocal and exp2 behind the FP64 rates, at the edges of their
tables' intervals."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W
from test_gpu_step import gpu_species, oracle_species

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
def test_rates_f64_interval_edges(ulps):
    """Fields at and beside every mantissa interval's ends, 2^-3 to 2^20 GV/m.  1e-12 relative
    (the FP64 form's bar) wherever no term of the exponent exceeds 400: each is
    off by 400 ln 2 2^-52 = 6e-14 at most, on either side."""
    sd = W.krypton_like()
    base = np.concatenate([2.0 ** k * (1 + np.arange(128) / 128.0) for k in range(-3, 20)])
    E = base.copy()
    for _ in range(abs(ulps)):
        E = np.nextafter(E, np.inf if ulps > 0 else 0.0)
    got = ionize.rates(gpu_species(sd), torch.tensor(E, device="cuda"), 0, sd.Z).cpu().numpy()
    ref = oracle.rates(oracle_species(sd), E, 0, sd.Z)
    big = ref > 2.0 ** -380
    assert big.sum() > 1000
    assert np.all(np.abs(got[big] - ref[big]) <= 1e-12 * ref[big])
