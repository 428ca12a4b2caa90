"""Which kernels a call runs on (csrc/xc_route.h), compiled for the host: the rules need sizes only."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_09803_gb300", "csrc")
DOPPLER, LORENTZ, W4, GH_BINNED, GH_SAMPLED, DOPPLER_BINNED, LORENTZ_BINNED, VV = range(8)

SHIM = """
#include "xc_route.h"
extern "C" int blocks64(int profile, double nu_A, double step, long long n_pts, double cutoff, unsigned long long n) {
    return xc::route_blocks64(profile, xc_grid{nu_A, step, (int64_t)n_pts}, cutoff, (size_t)n);
}
// 0: tiled kernels, 1: the same with far wings on the tensor cores, 2: blocks, 3: both rules at once (a fault)
extern "C" int route32(int profile, int flags, double cutoff, double width_mult, double step, long long n_pts,
                       unsigned long long n_lines, int n_cond, int allow_tc, int tiled) {
    const xc_grid g{1000.0, step, (int64_t)n_pts};
    xc_condition c{};
    c.T = 1000.0, c.P = 0.1, c.mass_da = 18.0, c.T_ref = 296.0, c.P_ref = 1.0, c.gamma_scale = 1.0;
    const xc::Route32 r{profile, flags, 20, cutoff, width_mult, xc::route_cut_steps(cutoff, width_mult, g, &c, 1), g,
                        (size_t)n_lines, (double)n_lines, n_cond, allow_tc != 0, tiled != 0};
    return 2 * xc::route_blocks32(r) + xc::route_tc32(r);
}
extern "C" int adjoint_blocks(int profile, double cutoff, double width_mult, double step, long long n_pts,
                              unsigned long long n_lines, int n_cond) {
    const xc_grid g{1000.0, step, (int64_t)n_pts};
    xc_condition c{};
    c.T = 1000.0, c.P = 0.1, c.mass_da = 18.0, c.T_ref = 296.0, c.P_ref = 1.0, c.gamma_scale = 1.0;
    return xc::route_adjoint_blocks(profile, 20, cutoff, xc::route_cut_steps(cutoff, width_mult, g, &c, 1), g,
                                    (double)n_lines, n_cond);
}
extern "C" double reach(unsigned long long n, double lo, double hi, double nu_A, double step, long long n_pts, double cutoff) {
    return xc::route_reach((size_t)n, lo, hi, xc_grid{nu_A, step, (int64_t)n_pts}, cutoff);
}
"""


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("route")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, str(d / "shim.cpp"), "-o", str(d / "r.so")],
                   check=True)
    L = C.CDLL(str(d / "r.so"))
    L.blocks64.argtypes = [C.c_int, C.c_double, C.c_double, C.c_longlong, C.c_double, C.c_ulonglong]
    L.route32.argtypes = [C.c_int, C.c_int, C.c_double, C.c_double, C.c_double, C.c_longlong, C.c_ulonglong, C.c_int,
                          C.c_int, C.c_int]
    L.reach.argtypes = [C.c_ulonglong, C.c_double, C.c_double, C.c_double, C.c_double, C.c_longlong, C.c_double]
    L.reach.restype = C.c_double
    L.adjoint_blocks.argtypes = [C.c_int, C.c_double, C.c_double, C.c_double, C.c_longlong, C.c_ulonglong, C.c_int]
    return L


TILED, TC, BLOCKS = 0, 1, 2


def r32(route, profile=W4, cut=2500.0, wm=0.0, n_pts=1_000_001, n=10_000_000, nc=32, flags=0, allow=1, tiled=0):
    r = route.route32(profile, flags, cut * 0.01, wm, 0.01, n_pts, n, nc, allow, tiled)
    assert r != 3
    return r


def test_what_the_blocks_do_not_take_keeps_the_tensor_cores(route):
    """Every reason that keeps a call from the blocks leaves its far wings on the tensor cores."""
    assert r32(route) == BLOCKS
    for kw in (dict(n=3 << 29), dict(n=(3 << 29) + 5, cut=500.0), dict(cut=2.0 ** 20), dict(cut=2.0 ** 21, n=1000, n_pts=4001),
               dict(tiled=1), dict(n=3000)):
        assert r32(route, **kw) == TC, kw
        assert r32(route, nc=15, **{**kw, "tiled": 1}) == TILED
        assert r32(route, flags=1, **{**kw, "tiled": 1}) == TILED
        assert r32(route, wm=500.0, **{**kw, "tiled": 1}) == TILED
        assert r32(route, allow=0, **{**kw, "tiled": 1}) == TILED
    assert r32(route, n_pts=1 << 30) == TILED        # the tensor-core form itself ends at 2^23 points
    assert r32(route, profile=VV) == TILED


def test_fp64_blocks_take_ordinary_grids(route):
    for nu_A, step, n in ((1000.0, 0.01, 200_001), (0.0, 0.01, 1_000_001), (20000.0, 1e-4, 1001), (-5.0, 0.01, 11)):
        assert route.blocks64(W4, nu_A, step, n, min(25.0, 1e5 * step), 100_000)
    assert not route.blocks64(VV, 1000.0, 0.01, 1001, 25.0, 1000)
    assert not route.blocks64(W4, 1000.0, 0.01, 1001, 25.0, 1 << 30)
    assert not route.blocks64(W4, 1000.0, 0.01, 1 << 30, 25.0, 1000)
    assert not route.blocks64(W4, 1000.0, 0.01, 1001, 0.01 * 2 ** 20, 1000)


def test_fp64_blocks_leave_steps_near_the_rounding_of_the_wavenumber(route):
    """The first-order term that follows a point's rounding is good to 3 (r / d)^2: every grid that is
    taken keeps it below 2.3e-16 at the nearest distance of a block, 60 steps."""
    taken = 0
    for nu in 10.0 ** np.arange(-2, 6):
        for step in 10.0 ** np.arange(-30.0, 2.0):
            r = np.spacing(nu) / 2 / step
            if route.blocks64(W4, nu, step, 1000, 1000 * step, 1000):
                taken += 1
                assert 3 * (r / 60.0) ** 2 < 2.3e-16, (nu, step)
            else:   # not a line further than it need be
                assert r > 2.0 ** -23, (nu, step)
    assert taken > 40


# measured on both sides of the rule (us, blocks and tiled): the faster form is the one chosen
MEASURED = [
    # profile, points, lines a point, cut (steps), width multiple, conditions, blocks, tiled
    (LORENTZ, 1000001, 0.003, 2500, 0, 12, 1696.4, 300.4),
    (LORENTZ, 1000001, 0.3, 256, 0, 6, 1001.1, 691.5),
    (LORENTZ, 1000001, 0.003, 256, 0, 2, 344.9, 142.7),
    (LORENTZ, 100001, 0.3, 256, 500, 12, 855.6, 1361.1),
    (LORENTZ, 1000001, 0.3, 2500, 0, 12, 2182.7, 4294.7),
    (LORENTZ, 100001, 0.3, 2500, 500, 1, 127.1, 189.4),
    (W4, 1000001, 0.03, 2500, 0, 12, 1568.3, 1106.8),
    (W4, 1000001, 0.03, 50, 0, 6, 853.9, 423.1),
    (W4, 1000001, 0.03, 50, 0, 4, 573.9, 349.2),
    (W4, 100001, 0.03, 256, 500, 1, 105.3, 152.3),
    (W4, 100001, 0.003, 256, 500, 4, 283, 421.9),
    (W4, 1000001, 0.3, 256, 500, 2, 656, 1425.5),
    (GH_BINNED, 1000001, 0.003, 50, 0, 6, 864.1, 357.1),
    (GH_BINNED, 1000001, 0.003, 50, 0, 1, 208.3, 147.6),
    (GH_BINNED, 1000001, 0.003, 256, 0, 6, 869.7, 481),
    (GH_BINNED, 1000001, 0.03, 2500, 500, 1, 263.4, 944.9),
    (GH_BINNED, 1000001, 0.3, 256, 500, 1, 1055, 3129.9),
    (GH_BINNED, 1000001, 0.03, 256, 0, 1, 243.8, 477.7),
    (GH_SAMPLED, 1000001, 0.003, 256, 500, 6, 1071.2, 726.4),
    (GH_SAMPLED, 1000001, 0.003, 50, 0, 6, 860.3, 250.5),
    (GH_SAMPLED, 1000001, 0.03, 50, 0, 6, 871, 460),
    (GH_SAMPLED, 100001, 0.03, 2500, 0, 1, 108.8, 498.9),
    (GH_SAMPLED, 1000001, 0.03, 2500, 0, 1, 265.2, 982.5),
    (GH_SAMPLED, 100001, 0.3, 256, 500, 1, 160.3, 434.9),
    (DOPPLER_BINNED, 1000001, 0.03, 2500, 0, 6, 168.1, 3163.1),
    (DOPPLER_BINNED, 100001, 0.003, 50, 0, 1, 70, 95.9),
    (DOPPLER_BINNED, 1000001, 0.03, 256, 0, 1, 84.6, 205.2),
    (LORENTZ_BINNED, 1000001, 0.003, 50, 0, 2, 334.2, 148.7),
    (LORENTZ_BINNED, 1000001, 0.003, 256, 0, 2, 339.3, 150),
    (LORENTZ_BINNED, 1000001, 0.03, 256, 0, 4, 604.3, 279.7),
    (LORENTZ_BINNED, 100001, 0.03, 2500, 0, 2, 112.4, 520.9),
    (LORENTZ_BINNED, 100001, 0.3, 2500, 500, 6, 545.1, 1304.7),
    (LORENTZ_BINNED, 100001, 0.03, 256, 500, 24, 1446.2, 1968.3),
]


@pytest.mark.parametrize("row", MEASURED)
def test_sparse_lists_run_the_faster_form(route, row):
    profile, n_pts, density, cut, wm, nc, blocks, tiled = row
    got = r32(route, profile=profile, cut=cut, wm=wm, n_pts=n_pts, n=max(2, int(n_pts * density)), nc=nc)
    assert (got == BLOCKS) == (blocks < tiled), (got, row)


# the adjoint: us with the block nodes and point by point
MEASURED_ADJOINT = [
    (LORENTZ, 1000001, 0.003, 256, 0, 6, 723.4, 230),
    (LORENTZ, 1000001, 0.003, 2500, 500, 3, 470.6, 223.3),
    (LORENTZ, 1000001, 0.3, 50, 0, 6, 1666, 1011.5),
    (LORENTZ, 100001, 0.003, 50, 0, 24, 440.6, 217.3),
    (LORENTZ, 1000001, 0.3, 2500, 0, 1, 952.6, 1381.1),
    (LORENTZ, 100001, 0.3, 2500, 0, 6, 575.2, 842.2),
    (W4, 100001, 0.003, 256, 0, 24, 502.3, 326.9),
    (W4, 1000001, 0.003, 50, 0, 3, 461, 216.6),
    (W4, 100001, 0.03, 256, 0, 24, 556.1, 410.8),
    (W4, 1000001, 0.003, 256, 0, 24, 2438.3, 678.7),
    (W4, 1000001, 0.03, 2500, 0, 1, 382, 631.8),
    (W4, 100001, 0.03, 2500, 0, 24, 629.9, 1590.9),
    (W4, 100001, 0.3, 2500, 0, 6, 702.9, 2423.4),
    (W4, 100001, 0.03, 2500, 0, 3, 252.4, 368),
    (GH_BINNED, 1000001, 0.003, 50, 0, 6, 797.2, 264.1),
    (GH_BINNED, 100001, 0.003, 50, 0, 6, 283.4, 205.3),
    (GH_BINNED, 1000001, 0.003, 256, 0, 6, 918.7, 466.8),
    (GH_BINNED, 1000001, 0.003, 50, 0, 1, 293.1, 196.7),
    (GH_BINNED, 100001, 0.3, 2500, 0, 1, 810.6, 3668.3),
    (GH_BINNED, 100001, 0.03, 2500, 0, 3, 466.5, 1494),
    (GH_BINNED, 100001, 0.003, 2500, 0, 6, 473.1, 1168.5),
    (GH_BINNED, 1000001, 0.03, 2500, 500, 1, 717.6, 1029.8),
]


@pytest.mark.parametrize("row", MEASURED_ADJOINT)
def test_sparse_adjoints_run_the_faster_form(route, row):
    profile, n_pts, density, cut, wm, nc, blocks, points = row
    got = route.adjoint_blocks(profile, cut * 0.01, wm, 0.01, n_pts, max(2, int(n_pts * density)), nc)
    assert bool(got) == (blocks < points), row


def test_adjoint_blocks_keep_their_limits(route):
    assert route.adjoint_blocks(W4, 25.0, 0.0, 0.01, 200_001, 300_000, 4)
    assert not route.adjoint_blocks(DOPPLER, 25.0, 0.0, 0.01, 200_001, 300_000, 4)
    assert not route.adjoint_blocks(W4, 25.0, 0.0, 0.01, 1 << 30, 1 << 30, 4)
    assert not route.adjoint_blocks(W4, 0.01 * 2 ** 20, 0.0, 0.01, 200_001, 300_000, 4)


def test_lines_in_reach(route):
    r = route.reach
    assert r(1000, 0.0, 10_000.0, 5000.0, 0.01, 100_000, 0.0) == pytest.approx(100.0)
    assert r(1000, 0.0, 10_000.0, 5000.0, 0.01, 100_000, 500.0) == pytest.approx(200.0)
    assert r(1000, 0.0, 10_000.0, 9900.0, 0.01, 100_000, 25.0) == pytest.approx(12.5)
    assert r(1000, 100.0, 200.0, 0.0, 0.01, 100_000, 25.0) == 1000.0     # the grid covers the list
    assert r(1000, 100.0, 200.0, 500.0, 0.01, 1000, 25.0) == 0.0
    assert r(7, 100.0, 100.0, 50.0, 0.01, 10_000, 25.0) == 7.0           # one wavenumber
