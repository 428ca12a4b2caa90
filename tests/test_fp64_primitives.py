"""The FP64 exponential of the per-line kernels (csrc/xc_exp64.cuh), replayed in exact arithmetic with its own
table and constants, and the short arctangent of the FP32 Gauss-Hermite blocks.

The exponential is under every FP64 strength, width and partition function: 0.51 units in the last
place is the bound that the source states (a wrong low word of one of the 512 table entries costs up to half a
unit, a wrong digit far more)."""
import os
import re
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_09803_gb300", "csrc")
SRC = open(os.path.join(CSRC, "xc_exp64.cuh")).read()
TABLE = [(float(a), float(b)) for a, b in re.findall(r"\{(-?[\d.e+-]+), (-?[\d.e+-]+)\}", SRC)]
mpmath = pytest.importorskip("mpmath")
mpmath.mp.prec = 200


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # one rounding


def constants():
    f = SRC[SRC.index("double exp64(double x)"):]
    scale = float(re.search(r"fma\(x, ([\d.]+), magic\)", f).group(1))
    c1, c2 = (float(v) for v in re.findall(r"fma\(-kf, ([\d.e-]+), [xr]\)", f))
    return scale, c1, c2


def exp64(x, scale, c1, c2):
    magic = 6755399441055744.0
    kd = fma(x, scale, magic)
    kf = kd - magic
    k = int(kf)
    r = fma(-kf, c2, fma(-kf, c1, x))
    q = fma(fma(r, 1.0 / 24.0, 1.0 / 6.0), r, 0.5)
    p = fma(r * r, q, r)
    hi, lo = TABLE[k % 512]
    return np.ldexp(hi + fma(hi, p, lo), k // 512)


def ulps(got, x):
    ref = mpmath.exp(mpmath.mpf(float(x)))
    return abs(mpmath.mpf(float(got)) - ref) / mpmath.mpf(float(np.spacing(float(ref))))


def test_table_of_powers():
    assert len(TABLE) == 512
    for j, (hi, lo) in enumerate(TABLE):
        ref = mpmath.mpf(2) ** (mpmath.mpf(j) / 512)
        assert hi == float(ref)
        assert abs(mpmath.mpf(hi) + mpmath.mpf(lo) - ref) < mpmath.mpf(2) ** -105, j


def test_exp64_within_its_bound():
    c = constants()
    rng = np.random.default_rng(1)
    j = np.arange(512)
    half = np.log(2.0) / 1024
    # every table entry at the middle and near both ends of its interval; the ends of the range; Boltzmann
    # factors and small arguments
    x = np.concatenate([j * np.log(2.0) / 512, (j + 0.499) * np.log(2.0) / 512, -(j + 0.4999) * np.log(2.0) / 512,
                        [0.0, -0.0, half, -half, 707.9999, -707.9999, 1e-300, -1e-17, 1e-9],
                        rng.uniform(-707.99, 707.99, 1500), -10.0 ** rng.uniform(-12, 2.8, 1500)])
    worst = max(ulps(exp64(float(v), *c), v) for v in x)
    assert worst < 0.51, worst


def test_short_arctangent():
    """gh_far_value: atan(t) = t - t^3/3 + t^5/5 up to kGhFarT, the rest below t^6/7 of it; what FP32 adds is
    its own rounding."""
    src = open(os.path.join(CSRC, "xc_f32.cuh")).read()
    top = float(re.search(r"kGhFarT = ([\d.]+)f", src).group(1))
    assert "fmaf(q, fmaf(q, 0.2f, -1.f / 3.f), 1.f)" in src
    t = np.linspace(1e-6, top, 4001)
    q = t * t
    assert np.max(np.abs(t * (1 + q * (-1 / 3 + 0.2 * q)) / np.arctan(t) - 1)) < 1.1e-10
    t32 = t.astype(np.float32)
    q32 = t32 * t32
    v = t32 * (np.float32(1) + q32 * (np.float32(-1 / 3) + np.float32(0.2) * q32))
    assert np.max(np.abs(v.astype(np.float64) / np.arctan(t32.astype(np.float64)) - 1)) < 3 * 2.0 ** -24
