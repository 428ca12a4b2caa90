"""Lines whose integer grid position lies beyond 2^30, on grids of about 2^30 points.

Their cuts reach back onto the grid, so the last points must equal a small grid that starts
there.  Positions are good to 1.8e-12 cm^-1 / step = 1.8e-7 steps on both sides and the profiles
(Doppler widths above 1000 steps) change by at most 1.6e-3 of their value a step: 6e-10, bound
1e-8 in FP64; FP32 2e-5 as between any two FP32 paths."""
import numpy as np
import pytest

import xcsynth as xs
from test_gpu_parity import eng, xc  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEP, NU_A, CUT = 1e-5, 100.0, 0.025
BEYOND = np.array([-3000.25, -900.4, -2.3, 41.7, 500.3, 1900.6, 2300.8])   # line positions from 2^30, in steps
TAIL = 4096


def setup(eng, n):  # noqa: F811
    L = xs.gen_lines(308, 0, len(BEYOND), 5000.0, 6000.0)
    L["nu"] = NU_A + (float(1 << 30) + BEYOND) * STEP
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(308, 200))
    return NU_A + (n - TAIL) * STEP


# the FP64 blocks, the FP32 blocks, and the tiled FP32 kernels (2^30 points and more)
@pytest.mark.parametrize("precision,n,tol", [("fp64", (1 << 30) - 1, 1e-8), ("fp32", (1 << 30) - 1, 2e-5),
                                             ("fp32", (1 << 30) + 1024, 2e-5)])
def test_lines_beyond_2_to_30(eng, xc, precision, n, tol):  # noqa: F811
    start = setup(eng, n)
    cond, opts = [xc.make_condition(300.0, 1e-2)], xc.make_opts("voigt_w4", precision, CUT)
    out = torch.empty((1, n), dtype=torch.float64, device="cuda:0")
    eng.cross_section_batched(cond, xc.make_grid(NU_A, STEP, n), opts, out)
    got = out[0, n - TAIL:].cpu().numpy()
    ref = eng.cross_section_batched(cond, xc.make_grid(start, STEP, TAIL), opts)[0]
    assert np.count_nonzero(ref) > 3000
    assert np.max(np.abs(got - ref) / np.maximum(ref, 1e-6 * ref.max())) < tol


def test_adjoint_of_lines_beyond_2_to_30(eng, xc):  # noqa: F811
    n = (1 << 30) + 1024
    start = setup(eng, n)
    cond, opts = [xc.make_condition(300.0, 1e-2)], xc.make_opts("voigt_w4", "fp32", CUT)
    w = torch.zeros((1, n), dtype=torch.float64, device="cuda:0")
    wt = 1e22 * np.random.default_rng(1).uniform(0.5, 1.5, TAIL)
    w[0, n - TAIL:] = torch.as_tensor(wt, device="cuda:0")
    got = eng.cross_section_vjp(cond, xc.make_grid(NU_A, STEP, n), opts, w)
    ref = eng.cross_section_vjp(cond, xc.make_grid(start, STEP, TAIL), xc.make_opts("voigt_w4", "fp64", CUT), wt[None])
    for k in ("dT", "dP", "d_gamma_ref_line", "d_n_line"):
        a, b = got[k].cpu().numpy() if hasattr(got[k], "cpu") else np.asarray(got[k]), np.asarray(ref[k])
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b)), k
