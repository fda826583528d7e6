"""ion_mlp_standardize: the moments' integer sums against wide sums, with columns inside
and outside the range they serve."""
import numpy as np
import pytest
import torch

from paper_2202_10647_gb300 import ionize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5000, 16384, 70001])
def test_moments_columns(n):
    """Mean within 1e-13 of the largest value (n additions of 2^-53 of it, taken 32 exactly and
    the rest pairwise), scale within 1e-12; a column of infinities or NaN leaves the
    others alone."""
    rng = np.random.default_rng(n)
    z = rng.normal(size=n)
    spike = z * 1e-3
    spike[n // 3] = 1e6
    cols = [z, z - z.mean(), 10.0 ** rng.uniform(-10, 10, n), spike, np.where(z > 0, 1.0, -1.0),
            z * 2.0 ** 395, z * 2.0 ** 410, z * 2.0 ** -395, z * 2.0 ** -420 + 0.0,
            np.full(n, 1.0 + 2.0 ** -52), 2.0 ** 30 + z * 2.0 ** -20, np.zeros(n)]
    Y = np.stack(cols + [z.copy(), z.copy()], 1)
    Y[n // 2, -2] = np.inf
    Y[n // 2, -1] = np.nan
    mean, scale, _ = ionize.mlp_standardize(torch.tensor(Y, device="cuda"), 1e-200)
    m, s = mean.cpu().numpy(), scale.cpu().numpy()
    k = len(cols)
    L = Y[:, :k].astype(np.longdouble)
    big = np.abs(Y[:, :k]).max(0)
    rm = L.mean(0)
    rs = np.maximum(np.sqrt(((L - rm) ** 2).sum(0) / (n - 1)), 1e-200)
    assert np.all(np.abs(m[:k] - rm) <= 1e-13 * big)
    assert np.all(np.abs(s[:k] - rs) <= 1e-12 * rs + 1e-13 * big)
    assert np.isinf(m[-2]) and np.isnan(m[-1])
