"""ion_mlp_standardize: columns whose spread is small beside their values."""
import numpy as np
import pytest
import torch

from paper_2202_10647_gb300 import ionize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5000, 70_001])
@pytest.mark.parametrize("ratio", [10, 20, 30, 40, 50])
def test_scale_of_offset_columns(n, ratio):
    """Offset 2^ratio times the spread.  Roundings of d = 2^-53 of the offset each: a slice's
    mean takes 23 (a thread's sum, 21 additions over 85 rows, the division), the column's 10
    more (a product, 8 additions, the division).  The squared deviations are summed about the
    rounded means: the variance is off by their errors squared, and by twice their errors times a
    slice mean's distance from the column's."""
    rng = np.random.default_rng(n + ratio)
    z = rng.normal(size=n)
    cols = [s * (2.0 ** e + z * 2.0 ** (e - ratio)) for s, e in ((1, 30), (-1, 3), (1, -200))]
    Y = np.stack(cols, 1)
    mean, scale, T = ionize.mlp_standardize(torch.tensor(Y, device="cuda"), 1e-300)
    L = Y.astype(np.longdouble)
    rm = L.mean(0)
    var = ((L - rm) ** 2).sum(0) / (n - 1)
    d = np.abs(Y).max(0) * 2.0 ** -53
    rows = 256 // 3 * 32
    far = np.max([np.abs(L[i:i + rows].mean(0) - rm) for i in range(0, n, rows)], 0)
    ds, dm = 23 * d, 33 * d
    tol = 2e-12 * var + 2 * (ds * ds + dm * dm + 2 * (ds + dm) * (far + dm))
    s = scale.cpu().numpy().astype(np.longdouble)
    assert np.all(np.abs(s * s - var) <= tol)
    assert np.all(np.abs(mean.cpu().numpy() - rm) <= dm)
    if ratio < 40:
        assert np.all(tol < 0.01 * var)


@pytest.mark.parametrize("value", [1.0 + 2.0 ** -52, -3.7e100, 1.0 / 3.0])
def test_scale_of_constant_columns(value):
    """No spread: the scale is the rounding of the mean at most."""
    Y = torch.full((40_003, 5), value, dtype=torch.float64, device="cuda")
    mean, scale, _ = ionize.mlp_standardize(Y, 1e-300)
    d = abs(value) * 2.0 ** -53
    assert float((mean - value).abs().max()) <= 33 * d
    assert float(scale.max()) <= 2 * 33 * d
