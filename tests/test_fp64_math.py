"""The fixed-point log2, 1/E, exp2 and e^z of csrc/fp64_math.cuh, their integer
steps restated here over the tables and constants of the source, against
mpmath: the errors that the source states."""
import os
import random
import re
import struct

import pytest
from mpmath import mp, mpf

from paper_2202_10647_gb300 import build

SRC = open(os.path.join(build.CSRC, "fp64_math.cuh")).read()
M32, M64 = 0xFFFFFFFF, (1 << 64) - 1


def numbers(name):
    body = re.search(name + r"\[\d+\] = \{(.*?)\};", SRC, re.S).group(1)
    return [int(x, 16) for x in re.findall(r"0x([0-9a-f]+)u", body)]


def constant(name):
    return int(re.search(name + r" = 0x([0-9a-f]+)u", SRC).group(1), 16)


LOG = numbers("kLogTab")
LOG = list(zip(LOG[0::2], LOG[1::2]))
EXP = numbers("kExpTab")
kLog = [constant(f"kLog{i}") for i in range(1, 7)]
kExp = [constant(f"kExp{i}") for i in range(1, 5)]
kLog2E = constant("kLog2E")


def words(x):
    b = struct.unpack(">Q", struct.pack(">d", x))[0]
    return b >> 32, b & M32


def double(bits):
    return struct.unpack(">d", struct.pack(">Q", bits & M64))[0]


def f32(x):
    return struct.unpack(">f", struct.pack(">f", x))[0]


def umulhi(a, b):
    return (a * b) >> 32


def mul_hi64(a, b):
    return ((a >> 32) * (b >> 32) + umulhi(a >> 32, b & M32) + umulhi(a & M32, b >> 32)) & M64


def mul_hi_short(S, a, bh, bl):
    return (((a & M32) * bh >> 32) + (a >> 32) * bh + (umulhi(a >> S & M32, bl) >> (32 - S))) & M64


def log2_f64(E):
    h, l = words(E)
    log, c = LOG[(h >> 13) & 127]
    m = (((h & 0xFFFFF) | 0x100000) << 32 | l) << 11
    mc = (m >> 32) * c + umulhi(m & M32, c)
    rho = (mc << 8) & M64
    rh, rl = rho >> 32, rho & M32
    B = kLog[2] - umulhi(kLog[3] - umulhi(kLog[4] - umulhi(kLog[5], rh), rh), rh)
    q = kLog[0] - mul_hi_short(13, kLog[1] - mul_hi_short(6, B, rh, rl), rh, rl)
    f = ((log + mul_hi64(rho, q) + 16) >> 5) + 0x3FF0000000000000
    return float((h >> 20) - 1024) + double(f)  # one rounding


def rcp_f64(E, off):
    """off: ulps by which the FP32 reciprocal is off (the SFU's is within 1)."""
    h, l = words(E)
    mant = struct.unpack(">f", struct.pack(">I", 0x3F800000 | (h & 0xFFFFF) << 3 | l >> 29))[0]
    sb = struct.unpack(">I", struct.pack(">f", f32(1.0 / mant)))[0] + off
    sb = min(max(sb, 0x3F000000), 0x3F800000)
    S = ((sb & 0x7FFFFF) | 0x800000) << ((sb >> 23) - 126)
    d = -((l * S + ((((h & 0xFFFFF) | 0x100000) * S & M32) << 32)) & M64) & M64
    d -= (d >> 63) << 64  # signed
    dq = d >> 40
    t = (d >> 12) + ((dq * dq & M32) >> 8)
    q = ((S << 36) + ((S * (t >> 4)) >> 24)) & M64
    M = (q + 64) >> 7
    return double(M + ((1021 - ((h >> 20) - 1023)) << 52))


def exp2_fixed(Y, tiny):
    yh = Y >> 32
    yh -= (yh >> 31) << 32
    T = EXP[(yh >> 13) & 255]
    rho = (Y << 19) & M64
    rh, rl = rho >> 32, rho & M32
    B = kExp[1] + umulhi(kExp[2] + umulhi(kExp[3], rh), rh)
    q = kExp[0] + mul_hi_short(10, B, rh, rl)
    S = T + (mul_hi64(T, mul_hi64(rho, q)) << 4)
    v = double(((S + 512) >> 10) + (((yh >> 21) + 1022) << 52))
    return v * 2.0 ** -256 if tiny else v


def exp2_f64(y):
    tiny = y <= -1022
    if tiny:
        y = max(y, -1200.0) + 256.0
    h, l = words(min(y, 1000.0))
    s = 1032 - ((h >> 20) & 0x7FF)
    m = (((h & 0xFFFFF) | 0x100000) << 32 | l) << 11
    m = ((m >> s) + 1) >> 1 if s < 64 else 0
    return exp2_fixed(-m & M64 if y < 0 else m, tiny)


def exp_f64(z):
    h, l = words(z)
    h = min(h & 0x7FFFFFFF, 0x40875000)
    P = mul_hi64((((h & 0xFFFFF) | 0x100000) << 32 | l) << 11, kLog2E)
    s = 1032 - (h >> 20)
    if s:
        P = ((P >> (s - 1)) + 1) >> 1 if s < 65 else 0
    tiny = P >= 1022 << 53
    return exp2_fixed(-(P - (256 << 53 if tiny else 0)) & M64, tiny)


def ulps(got, ref):
    """Error in ulp of the result, in 2^-1074 below the normal range."""
    e = max(int(mp.floor(mp.log(abs(ref), 2))), -1022)
    return abs(mpf(got) - ref) / mpf(2) ** (e - 52)


@pytest.fixture(autouse=True)
def precision():
    with mp.workprec(113):
        yield


def fields(lo, hi, n):
    """Over the range, and beside the ends of every mantissa interval."""
    r = random.Random(7)
    x = [(1 + r.random()) * 2.0 ** r.randint(lo, hi - 1) for _ in range(n)]
    for j in range(128):
        e = 2.0 ** r.randint(lo, hi - 1) * (1 + j / 128)
        x += [e, double(words(e)[0] << 32 | words(e)[1] + 1), e * (1 - 2.0 ** -53)]
    return x


def test_log2():
    """In ulp of max(|log2 E|, 1): the fixed-point fraction is off by 0.57 units of 2^-52, and
    from 2 on the sum with the exponent rounds it."""
    for E in fields(-20, 60, 6000):
        ref = mp.log(mpf(E), 2)
        k = max(int(mp.floor(mp.log(abs(ref), 2))) if ref else 0, 0)
        bar = 0.57 if k == 0 else 0.5 + 0.57 / 2 ** k
        assert abs(mpf(log2_f64(E)) - ref) / mpf(2) ** (k - 52) <= bar


@pytest.mark.parametrize("off", [-1, 0, 1])
def test_reciprocal(off):
    for E in fields(-20, 60, 3000) + fields(-1000, 1000, 500):
        assert ulps(rcp_f64(E, off), 1 / mpf(E)) <= 0.56


def test_exp2():
    r = random.Random(3)
    for y in [r.uniform(-1000, 1000) for _ in range(4000)] + [r.uniform(-2, 2) for _ in range(1000)]:
        assert ulps(exp2_f64(y), mpf(2) ** mpf(y)) <= 0.97
    for y in [r.uniform(-1074, -1022) for _ in range(500)]:
        assert ulps(exp2_f64(y), mpf(2) ** mpf(y)) <= 1.5
    assert exp2_f64(-1076.0) == exp2_f64(-5e4) == 0.0
    assert exp2_f64(1000.0) == exp2_f64(2e4) == 2.0 ** 1000


def test_exp():
    r = random.Random(5)
    for lo, hi, bar in ((0, 256, 0.99), (256, 512, 1.2), (512, 708, 1.9), (709, 745, 1.5)):
        for _ in range(2000):
            z = -r.uniform(lo, hi)
            assert ulps(exp_f64(z), mp.exp(mpf(z))) <= bar
    for z in [-2.0 ** r.uniform(-60, 0) for _ in range(1000)]:
        assert ulps(exp_f64(z), mp.exp(mpf(z))) <= 0.99
    assert exp_f64(-0.0) == exp_f64(-1e-300) == 1.0
    assert exp_f64(-745.2) == exp_f64(-746.0) == exp_f64(-1e30) == 0.0
