"""ion_conservation in FP32 around its blocks of 1,024 cells and its groups of 8 planes,
with targets that are and are not floats, and one past the float range."""
import math

import numpy as np
import pytest
import torch

from paper_2202_10647_gb300 import ionize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 1023, 1024, 1025, 1028, 3077])
@pytest.mark.parametrize("planes", [1, 7, 8, 9, 17])
@pytest.mark.parametrize("target", [1.0, 0.1, -3.0, 1e35])
def test_conservation_tiles(n, planes, target):
    """The deviation is rounded to float two times at most (2^-23 of it); the float-float sums
    of `planes` terms below 1 are off by less than planes^2 2^-47."""
    rng = np.random.default_rng(n * 32 + planes)
    ld = (n + 3) // 4 * 4 + 4
    N = rng.uniform(0, 1, (planes, ld)).astype(np.float32)
    N[:, n:] = 100.0  # padding is not looked at
    want = max(abs(math.fsum([*map(float, N[:, c]), -target])) for c in range(n))
    out = torch.zeros(1, device="cuda")
    ionize.conservation(torch.tensor(N, device="cuda"), out, target=target, ncells=n)
    assert abs(float(out.cpu()) - want) <= 2.0 ** -23 * want + planes ** 2 * 2.0 ** -47
