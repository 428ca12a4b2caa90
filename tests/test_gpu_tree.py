"""The block-interpolated FP32 sweep against the general CUDA-core path (a fixed tile shape
selects it) and the oracle, at the edges of its blocks and over the forms it accepts.

Tolerances: against the oracle those of the FP32 path (2e-4 / band 1e-5); between the two
FP32 paths 2e-5 relative above 1e-6 of the peak, as between the other FP32 paths (two FP32
summation orders, interpolation error below 2e-8)."""
import numpy as np
import pytest

import xcsynth as xs
from test_gpu_parity import TOL32, TOL32_BAND, eng, metrics, oracle_sigma, xc  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROFILES = ["voigt_w4", "lorentz", "doppler", "doppler_binned", "lorentz_binned", "voigt_gh_binned", "voigt_gh_sampled"]


def both(eng, conds, grid, opts):  # noqa: F811
    got = eng.cross_section_batched(conds, grid, opts)
    assert "block-interpolated" in eng.tuning()
    eng.set_tile_shape(8, 1)
    try:
        ref = eng.cross_section_batched(conds, grid, opts)
        assert "block-interpolated" not in eng.tuning()
    finally:
        eng.set_tile_shape(0, 0)
    return got, ref


def close(got, ref):
    m = ref > 1e-6 * ref.max(axis=1, keepdims=True)
    return float(np.max(np.abs(got[m] - ref[m]) / ref[m])) if m.any() else 0.0


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 127, 513, 4097])
@pytest.mark.parametrize("profile", PROFILES)
def test_block_edges(eng, xc, profile, n):  # noqa: F811
    L = xs.gen_lines(301, 0, 3000, 1000.0, 1060.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(301, 500))
    conds = [xc.make_condition(T, P) for T, P in ((300.0, 1e-3), (900.0, 0.3), (2500.0, 10.0))]
    for nu_A, step, cut, wm in ((1010.0, 0.01, 25.0, 0.0), (1059.37, 0.0137, 3.0, 0.0), (990.0, 0.01, 25.0, 300.0)):
        got, ref = both(eng, conds, xc.make_grid(nu_A, step, n), xc.make_opts(profile, "fp32", cut, wm))
        assert np.all(np.isfinite(got))
        assert close(got, ref) < 2e-5, (profile, n, nu_A, cut, wm)
        assert np.all((got == 0) == (ref == 0)) or profile.startswith("doppler") or profile.endswith("binned")


@pytest.mark.parametrize("n_cond", [1, 3, 40])
def test_against_oracle_with_long_cut(eng, xc, oracle_lib, n_cond):  # noqa: F811
    """2500-step cut, all three block levels, a ragged grid past both ends of the list, threshold
    and emission; 40 conditions run on the blocks as well (a cut of 1024 steps or more)."""
    L = xs.gen_lines(302, 0, 20_000, 500.0, 600.0)
    E, g = xs.gen_states(302, 1000)
    eng.load_lines(L)
    eng.set_states(E, g)
    TP = [(300.0 * 1.06 ** i, 1e-3 * 1.27 ** i) for i in range(n_cond)]
    nu_A, step, n = 480.03, 0.01, 13_337
    for quantity, thr in (("absorption", None), ("emission", ("hitran", 550.0, 1e-24))):
        got = eng.cross_section_batched([xc.make_condition(T, P) for T, P in TP], xc.make_grid(nu_A, step, n),
                                        xc.make_opts("voigt_w4", "fp32", 25.0, quantity=quantity, threshold=thr))
        assert "block-interpolated" in eng.tuning()
        for i in {0, n_cond // 2, n_cond - 1}:
            ref = oracle_sigma(oracle_lib, L, E, g, *TP[i], nu_A, step, n, "voigt_w4", 25.0, quantity=quantity,
                               threshold=thr)
            mr, band = metrics(got[i], ref)
            assert mr < TOL32 and band < TOL32_BAND, (quantity, i, mr, band)


def test_hotter_conditions_after_cooler_ones(eng, xc):  # noqa: F811
    """The radii follow the call's own conditions: a hot call after a cold one of the same shape."""
    L = xs.gen_lines(303, 0, 4000, 1000.0, 1030.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(303, 500))
    grid, opts = xc.make_grid(1000.0, 0.01, 3001), xc.make_opts("voigt_w4", "fp32", 25.0)
    out = torch.zeros((1, 3001), dtype=torch.float64, device="cuda:0")
    eng.cross_section_batched([xc.make_condition(100.0, 0.01)], grid, opts, out)
    eng.cross_section_batched([xc.make_condition(3000.0, 0.01)], grid, opts, out)
    hot = out.cpu().numpy()
    _, ref = both(eng, [xc.make_condition(3000.0, 0.01)], grid, opts)
    assert close(hot, ref) < 2e-5


def test_hotter_conditions_in_a_replayed_graph(eng, xc):  # noqa: F811
    """The tiled sweep's centre zones in a graph captured for a cold call and replayed for a hot one."""
    L = xs.gen_lines(303, 0, 4000, 1000.0, 1030.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(303, 500))
    grid, opts = xc.make_grid(1000.0, 0.01, 3001), xc.make_opts("voigt_w4", "fp32", 25.0)
    out = torch.zeros((1, 3001), dtype=torch.float64, device="cuda:0")
    eng.set_tile_shape(8, 1)
    try:
        eng.cross_section_batched([xc.make_condition(100.0, 0.01)], grid, opts, out)
        eng.cross_section_batched([xc.make_condition(3000.0, 0.01)], grid, opts, out)
    finally:
        eng.set_tile_shape(0, 0)
    ref = eng.cross_section_batched([xc.make_condition(3000.0, 0.01)], grid, opts)
    assert close(out.cpu().numpy(), ref) < 2e-5


@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz"])
@pytest.mark.parametrize("n_lines", [3001, 40_001, 40_400, 100_001])
@pytest.mark.parametrize("n_cond", [5, 16])
def test_sparse_lists_on_large_outputs(eng, xc, n_cond, n_lines, profile):  # noqa: F811
    """Either side of the lines a point below which the tiled kernels run (200 and 500 pairs a point)."""
    L = xs.gen_lines(307, 0, n_lines, 990.0, 11010.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(307, 500))
    grid = xc.make_grid(1000.0, 0.01, 1_000_003)
    conds = [xc.make_condition(400.0 + 60.0 * i, 0.01 * 1.5 ** i) for i in range(n_cond)]
    got = eng.cross_section_batched(conds, grid, xc.make_opts(profile, "fp32", 25.0))
    for c in (0, n_cond - 1):
        ref = eng.cross_section_batched([conds[c]], grid, xc.make_opts(profile, "fp64", 25.0))
        assert close(got[c:c + 1], ref) < 2e-5


# ------------------------------------------------------------------ FP64
def binned64(L, Q, T, P, x, step, cut, wm, profile):
    """Binned profiles with one arctangent per node.  (The oracle takes the difference of two, which
    is off by 2e-11 for narrow lines far from the point: checked with 40 digits.)"""
    c2 = 6.62607015e-34 * 2.99792458e10 / 1.380649e-23
    nu, f = L["nu"], {k: v.astype(np.float64) for k, v in L.items()}
    al = nu * np.sqrt(2 * 1.380649e-23 * T * np.log(2) / (18 * 1.66053906660e-27)) / 2.99792458e8
    ga = f["gamma_ref"] * (296.0 / T) ** f["n_T"] * P
    S = f["g_up"] * f["A"] / (8 * np.pi * 2.99792458e10 * Q * nu ** 2) * np.exp(-c2 * f["elower"] / T)
    S = S * -np.expm1(-c2 * nu / T)
    c = np.minimum(cut, wm * np.maximum(al, ga)) if wm else np.full_like(nu, cut)
    xj, wj = np.polynomial.hermite.hermgauss(20) if profile == "voigt_gh_binned" else (np.zeros(1), np.full(1, np.pi ** 0.5))
    out = np.empty_like(x)
    for k, xk in enumerate(x):
        D = xk - nu
        d = D[:, None] - (al / np.sqrt(np.log(2)))[:, None] * xj
        v = np.arctan2(step * ga[:, None], (d + step / 2) * (d - step / 2) + ga[:, None] ** 2) @ wj
        out[k] = (S * v)[np.abs(D) <= c].sum() * np.pi ** -1.5 / step
    return out


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 513, 4097])
@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz", "voigt_gh_binned", "doppler", "lorentz_binned"])
def test_fp64_blocks_against_oracle(eng, xc, oracle_lib, profile, n):  # noqa: F811
    """FP64 blocks: 1e-12 of every value (the direct FP64 sum agreed with the oracle to 1.6e-13;
    interpolation error 1e-16, point positions to first order)."""
    L = xs.gen_lines(304, 0, 1500, 1000.0, 1060.0)
    E, g = xs.gen_states(304, 500)
    eng.load_lines(L)
    eng.set_states(E, g)
    for nu_A, step, cut, wm, T, P in ((1010.003, 0.01, 25.0, 0.0, 900.0, 0.3), (1059.37, 0.0137, 3.0, 0.0, 300.0, 1e-3),
                                      (990.0, 0.01, 25.0, 300.0, 2500.0, 10.0)):
        got = eng.cross_section(xc.make_condition(T, P), xc.make_grid(nu_A, step, n),
                                xc.make_opts(profile, "fp64", cut, wm))
        if profile.endswith("binned"):
            ref = binned64(L, oracle_lib.partition_function(E, g, T)[0], T, P, nu_A + np.arange(n) * step, step, cut, wm,
                           profile)
        else:
            ref = oracle_sigma(oracle_lib, L, E, g, T, P, nu_A, step, n, profile, cut, wm)
        assert metrics(got, ref)[0] < 1e-12, (profile, n, nu_A)


# ------------------------------------------------------------------ adjoint
@pytest.mark.parametrize("n", [1, 33, 65, 513, 5003])
@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz", "voigt_gh_binned"])   # Doppler takes no blocks
def test_adjoint_on_blocks_against_fp64(eng, xc, profile, n):  # noqa: F811
    """The FP32 adjoint (block nodes, both cut forms, lines off the grid, 3 conditions) against the
    FP64 adjoint, which sums every point; tolerance of the FP32 adjoint 1e-4 of the largest line."""
    L = xs.gen_lines(305, 0, 1200, 1000.0, 1070.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(305, 500))
    conds = [xc.make_condition(T, P) for T, P in ((500.0, 0.01), (900.0, 0.5), (1600.0, 4.0))]
    rng = np.random.default_rng(n)
    w = 1e22 * rng.uniform(0.5, 1.5, (3, n))
    for nu_A, step, cut, wm in ((1020.0, 0.01, 25.0, 0.0), (1055.5, 0.0137, 4.0, 0.0), (1010.0, 0.01, 25.0, 400.0)):
        grid = xc.make_grid(nu_A, step, n)
        r32 = eng.cross_section_vjp(conds, grid, xc.make_opts(profile, "fp32", cut, wm), w)
        r64 = eng.cross_section_vjp(conds, grid, xc.make_opts(profile, "fp64", cut, wm), w)
        for k in ("dT", "dP", "d_gamma_ref_line", "d_n_line"):
            a, b = np.asarray(r32[k]), np.asarray(r64[k])
            assert np.max(np.abs(a - b)) <= 1e-4 * max(np.max(np.abs(b)), 1e-300), (k, profile, n, nu_A)


# ------------------------------------------------------------------ sort
@pytest.mark.parametrize("case", ["dense", "runs", "long_run", "two", "narrow"])
def test_sort_of_lines_that_agree_in_their_high_digits(eng, xc, case):  # noqa: F811
    """The in-place finish of the sort: many short runs of nearly equal wavenumbers, a run that is
    too long for it, equal wavenumbers (input order), and keys whose low digits alone differ."""
    rng = np.random.default_rng(7)
    n = {"two": 2}.get(case, 50_000)
    L = xs.gen_lines(306, 0, n, 1.0, 9000.0)
    base = L["nu"].copy()
    if case in ("runs", "long_run"):
        L["nu"] = np.repeat(base[::10], 10)[:n] * (1.0 + rng.integers(0, 40, n) * 2.0 ** -50)
    if case == "long_run":
        L["nu"][1000:2000] = 5000.0 + rng.integers(0, 300, 1000) * 2.0 ** -40
    if case == "narrow":
        L["nu"] = 4000.0 + rng.integers(0, 5000, n) * 2.0 ** -40
    p = rng.permutation(n)
    L = {k: v[p] for k, v in L.items()}
    eng.load_lines(L)
    order = np.argsort(L["nu"], kind="stable")
    assert np.array_equal(eng.get_permutation(), order.astype(np.uint32))
    got = eng.get_lines()
    for k in L:
        assert np.array_equal(got[k], L[k][order]), (case, k)
