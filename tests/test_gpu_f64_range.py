"""ion_rates in FP64 over every field it takes, and down to rates below the
normal range, against Eq. 1 in 40 digits."""
import math

import numpy as np
import pytest
import torch
from mpmath import mp, mpf

from paper_2202_10647_gb300 import ionize, workloads as W

pytestmark = pytest.mark.gpu


def table(sd, omega):
    """a, b, C of log2 W_k [1/fs] = a - b log2|E| - C/|E| (E_a = 510 GV/m, U_H = 13.6 eV)."""
    f = math.factorial
    for k, (U, l, m) in enumerate(zip(sd.U, sd.l, sd.m)):
        Q, am = mpf(k + 1), abs(m)
        ns = Q * mp.sqrt(mpf(13.6) / mpf(U))
        flm = mpf((2 * l + 1) * f(l + am)) / (2 ** am * f(am) * f(l - am))
        x = 2 * ns - am - 1
        lg = (mp.log(mpf(omega) * mpf(10) ** -15) + mp.log(3 * ns ** 3 / (mp.pi * Q ** 3)) / 2
              + mp.log(Q * Q / (2 * ns * ns)) + 2 * ns * mp.log(2 * mp.e / ns)
              + mp.log(flm / (2 * mp.pi * ns)) + x * mp.log(2 * Q ** 3 / ns ** 3))
        b = x - mpf(1) / 2
        yield lg / mp.log(2) + b * mp.log(510, 2), b, 2 * Q ** 3 / (3 * ns ** 3) * 510 / mp.log(2)


@pytest.mark.parametrize("omega", [4.13e16, 4.13e-10])
def test_rates_f64_over_all_fields(omega):
    """|E| from just above 1e-6 (where Eq. 1 ends) to 1.7e308, with the usual prefactor and
    with one that puts the cutoff's rates below 2^-1022.  Bar: 8 roundings of the largest term
    of the exponent (the table's own among them), and two units of 2^-1074; 0 past the
    cutoff and at 1e-6, 2^1000 at most."""
    sd = W.krypton_like()
    sp = ionize.Species(sd.U, sd.l, sd.m, (omega, 510.0, 13.6))
    r = np.random.default_rng(1)
    E = np.concatenate([10.0 ** r.uniform(-5.99, 308.0, 300), 10.0 ** r.uniform(-1, 6, 900),
                        [1.0001e-6, 1e-6, 2.0 ** 1019.5, 2.0 ** 1020.5, 1.7e308]])
    got = ionize.rates(sp, torch.tensor(E, device="cuda"), 0, sd.Z).cpu().numpy()
    small = 0
    with mp.workdps(40):
        lE = [mp.log(mpf(float(e)), 2) for e in E]
        for k, (a, b, C) in enumerate(table(sd, omega)):
            cut = mpf(700) / mp.log(2)
            for i, e in enumerate(E):
                q = C / mpf(float(e))
                if abs(q / cut - 1) < 1e-12:
                    continue
                if q > cut or e <= 1e-6:
                    assert got[k, i] == 0.0
                    continue
                y = a - b * lE[i] - q
                ref = mpf(2) ** min(y, 1000)
                size = abs(a) + abs(b * lE[i]) + q
                tol = ref * 8 * size * mpf(2) ** -52 + 2 * mpf(2) ** -1074 + ref * mpf(2) ** -51
                assert abs(mpf(float(got[k, i])) - ref) <= tol, (k, e)
                small += 0 < got[k, i] < 2.3e-308
    assert small > 50 or omega > 1
