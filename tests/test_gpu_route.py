"""Calls at the edges of the routing rules (csrc/xc_route.h), on the device."""
import numpy as np
import pytest

import xcsynth as xs
from test_gpu_parity import eng, metrics, xc  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1e-5, 1e-6, 1e-8, 1e-13, 1e-30])
def test_fp64_grids_of_fine_steps(eng, xc, oracle_lib, step):  # noqa: F811
    """From steps the blocks take down to steps below the rounding of the wavenumber, where all points
    coincide: 1e-12 of the oracle, as the FP64 paths elsewhere (both form nu_A + k step alike).  The
    oracle's point by point form: its sweep finds a line's range from floor((nu -+ cut - nu_A) / step) to
    within one point, which does not hold below the rounding."""
    nu_A, n = 10_000.0, 1500
    L = xs.gen_lines(309, 0, 40, 9000.0, 11000.0)
    rng = np.random.default_rng(309)
    L["nu"] = np.sort(np.concatenate([[nu_A], nu_A + rng.uniform(-600, 2100, 39) * step]))
    E, g = xs.gen_states(309, 200)
    eng.load_lines(L)
    eng.set_states(E, g)
    cut = 700.0 * step
    got = eng.cross_section(xc.make_condition(300.0, 1e-9), xc.make_grid(nu_A, step, n), xc.make_opts("voigt_w4", "fp64", cut))
    Q, dQ = oracle_lib.partition_function(E, g, 300.0)
    ref = oracle_lib.cross_section_points(L, oracle_lib.make_condition(300.0, 1e-9, Q, dQ), nu_A, step, np.arange(n),
                                          oracle_lib.make_opts("voigt_w4", cut), nthreads=4)
    assert metrics(got, ref)[0] < 1e-12


@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz"])
def test_adjoint_of_width_limited_cuts_under_a_mixture(eng, xc, profile):  # noqa: F811
    """The cut follows the mixture's width, not the list's own gamma_ref (here ten times it): FP32 adjoint
    against the FP64 one, 1e-4 of the largest as in the other adjoint tests."""
    L = xs.gen_lines(310, 0, 1500, 1000.0, 1060.0)
    L["gamma_ref"] *= np.float32(10.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(310, 500))
    eng.set_broadening([xc.make_broadener("constant", 0.7, 0.05, 0.6), xc.make_broadener("constant", 0.3, 0.09, 0.4)])
    conds = [xc.make_condition(T, P) for T, P in ((500.0, 0.2), (900.0, 1.0), (1600.0, 3.0))]
    n = 4001
    w = 1e22 * np.random.default_rng(310).uniform(0.5, 1.5, (3, n))
    grid = xc.make_grid(1010.0, 0.01, n)
    r32, r64 = (eng.cross_section_vjp_broadening(conds, grid, xc.make_opts(profile, p, 25.0, 100.0), w, 2)
                for p in ("fp32", "fp64"))
    eng.set_broadening([])
    for k in ("dT", "dP", "d_gamma_scale", "d_n_shift", "d_gamma0_broad", "d_n_broad"):
        a, b = np.asarray(r32[k]), np.asarray(r64[k])
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b)), k


def test_adjoint_of_more_conditions_than_a_grid_dimension(eng, xc):  # noqa: F811
    """65 536 conditions and more: each condition's gradients as in a call of its own (the FP32 sums of
    one condition do not depend on the others: equal)."""
    L = xs.gen_lines(311, 0, 3, 1000.0, 1001.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(311, 20))
    nc, n = 65_600, 130
    conds = [xc.make_condition(700.0, 0.1 + 1e-4 * i) for i in range(nc)]
    w = torch.full((nc, n), 1e22, dtype=torch.float64, device="cuda:0")
    grid, opts = xc.make_grid(1000.0, 0.01, n), xc.make_opts("voigt_w4", "fp32", 25.0)
    r = eng.cross_section_vjp(conds, grid, opts, w, per_line=False)
    for i in (0, 65_534, 65_535, 65_536, nc - 1):
        one = eng.cross_section_vjp([conds[i]], grid, opts, w[i:i + 1], per_line=False)
        assert float(r["dP"][i]) == float(one["dP"][0]) != 0.0 and float(r["dT"][i]) == float(one["dT"][0]), i


def with_room(room, f):
    """f() with `room` bytes left free on the device."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda:0")
    try:
        return f()
    finally:
        del fill
        torch.cuda.empty_cache()


def test_less_room_than_the_blocks_want(xc):
    """Where the constants of 14 conditions x 1e7 lines (4.5 GB) do not fit, the blocks take four
    conditions at a time (4, 4, 4, 2), then one, and the tiled kernels run what is left no room for."""
    n, nc = 10_000_000, 14
    grid, opts = xc.make_grid(1000.0, 0.01, 50_001), xc.make_opts("voigt_w4", "fp32", 25.0)
    conds = [xc.make_condition(400.0 + 150.0 * i, 0.01 * 1.6 ** i) for i in range(nc)]
    out = torch.empty((4, nc, 50_001), dtype=torch.float64, device="cuda:0")
    ran = []
    for i, room in enumerate((None, 3 << 30, 1 << 30, 320 << 20)):
        with xc.Engine(0) as e:
            e.load_lines(xs.gen_lines_torch(312, 0, n, 990.0, 1510.0, device="cuda:0"))
            e.set_states(*xs.gen_states(312, 500))
            call = lambda: e.cross_section_batched(conds, grid, opts, out[i])  # noqa: E731
            call() if room is None else with_room(room, call)
            ran.append(e.tuning())
    assert ["block-interpolated" in r for r in ran] == [True, True, True, False], ran
    assert [r.split(",")[-1].split()[0] for r in ran[:3]] == ["14", "4", "1"], ran
    for i in (1, 2, 3):
        ref = out[0]
        m = ref > 1e-6 * ref.amax(dim=1, keepdim=True)
        assert float(((out[i] - ref).abs() / ref)[m].max()) < 2e-5, i


def test_more_conditions_than_are_ordered(eng, xc):  # noqa: F811
    """Above 1024 conditions the sweep leaves them in the caller's order: 2e-5 of FP64."""
    eng.load_lines(xs.gen_lines(313, 0, 400, 1000.0, 1010.0))
    eng.set_states(*xs.gen_states(313, 100))
    conds = [xc.make_condition(300.0 + 2.0 * ((7 * i) % 1100), 0.01 + 0.001 * i) for i in range(1100)]
    grid = xc.make_grid(1001.0, 0.01, 777)
    got = eng.cross_section_batched(conds, grid, xc.make_opts("voigt_w4", "fp32", 25.0))
    assert "block-interpolated" in eng.tuning()
    for c in (0, 1, 550, 1023, 1024, 1099):
        ref = eng.cross_section_batched([conds[c]], grid, xc.make_opts("voigt_w4", "fp64", 25.0))[0]
        m = ref > 1e-6 * ref.max()
        assert np.max(np.abs(got[c] - ref)[m] / ref[m]) < 2e-5, c


@pytest.mark.parametrize("profile,sparse,dense", [("lorentz", 20_000, 500_000), ("lorentz_binned", 10_000, 200_000),
                                                  ("voigt_gh_sampled", 2_000, 100_000), ("voigt_w4", 10_000, 400_000)])
def test_sparse_and_dense_lists_run_their_own_kernels(eng, xc, profile, sparse, dense):  # noqa: F811
    """Either side of the rule for sparse lists, and both against the general path (a fixed tile shape),
    2e-5 as between any two FP32 paths.  (FP32 itself is 2.0e-5 from FP64 here: a Lorentz width of 0.07 steps
    at the sampled Gauss-Hermite nodes, blocks and tiled kernels alike.)"""
    grid = xc.make_grid(1000.0, 0.01, 500_003)
    conds = [xc.make_condition(400.0 + 90.0 * i, 0.01 * 1.9 ** i) for i in range(6)]
    opts = xc.make_opts(profile, "fp32", 5.0)
    eng.set_states(*xs.gen_states(314, 500))
    for n, blocks in ((sparse, False), (dense, True)):
        eng.load_lines(xs.gen_lines(314, 0, n, 995.0, 6005.0))
        got = eng.cross_section_batched(conds, grid, opts)
        assert ("block-interpolated" in eng.tuning()) == blocks, (profile, n, eng.tuning())
        eng.set_tile_shape(8, 1)
        ref = eng.cross_section_batched(conds, grid, opts)
        eng.set_tile_shape(0, 0)
        m = ref > 1e-6 * ref.max(axis=1, keepdims=True)
        assert np.max(np.abs(got - ref)[m] / ref[m]) < 2e-5, (profile, n)


@pytest.mark.parametrize("wm", [0.0, 400.0])
@pytest.mark.parametrize("profile,n_lines,n,blocks", [
    ("lorentz", 20_000, 5003, 1), ("lorentz", 300, 200_003, 0), ("voigt_w4", 20_000, 5003, 1),
    ("voigt_w4", 300, 200_003, 0), ("voigt_gh_binned", 8000, 2003, 1), ("voigt_gh_binned", 20, 200_003, 0)])
def test_adjoint_of_sparse_and_dense_lists(eng, xc, profile, n_lines, n, blocks, wm):  # noqa: F811
    """Block nodes and all points, fixed and width-limited cuts, against the FP64 adjoint (1e-4 of the
    largest, as in the other adjoint tests); the projection on the nodes is one launch more."""
    L = xs.gen_lines(315, 0, n_lines, 2995.0, 3005.0 + 0.01 * n)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(315, 500))
    conds = [xc.make_condition(T, P) for T, P in ((500.0, 0.01), (900.0, 0.5), (1600.0, 4.0))]
    w = 1e22 * np.random.default_rng(315).uniform(0.5, 1.5, (3, n))
    cut = 25.0 if blocks else 0.5
    grid = xc.make_grid(3000.0, 0.01, n)
    for _ in range(2):   # the handle's first call of a Gauss-Hermite profile also makes its nodes
        r32 = eng.cross_section_vjp(conds, grid, xc.make_opts(profile, "fp32", cut, wm), w)
    assert eng.last_launch_count() == 7 + blocks
    r64 = eng.cross_section_vjp(conds, grid, xc.make_opts(profile, "fp64", cut, wm), w)
    for k in ("dT", "dP", "d_gamma_ref_line", "d_n_line"):
        a, b = np.asarray(r32[k]), np.asarray(r64[k])
        assert np.max(np.abs(a - b)) <= 1e-4 * max(np.max(np.abs(b)), 1e-300), k


@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz", "lorentz_binned", "voigt_gh_binned", "doppler"])
@pytest.mark.parametrize("n_lines,cut", [(40, 2.0), (150, 4.0), (600, 8.0)])
def test_sparse_grid_shards_are_bit_exact(eng, xc, profile, n_lines, cut):  # noqa: F811
    """FP64 lists of 0 to a dozen lines a block, where blocks with few lines are left to the points: a shard
    of the grid that holds its own lines only decides alike (step 2^-7: exact points)."""
    from paper_1801_09803_gb300.shard import grid_shard, halo_line_range
    S = xs.gen_lines(316, 0, n_lines, 990.0, 1075.0)
    S = {k: v[np.argsort(S["nu"], kind="stable")] for k, v in S.items()}
    eng.set_states(*xs.gen_states(316, 300))
    nu_A, step, n, cond = 1000.0, 1.0 / 128.0, 8193, xc.make_condition(900.0, 0.3)
    opts = xc.make_opts(profile, "fp64", cut)
    eng.load_lines(S, assume_sorted=True)
    full = eng.cross_section(cond, xc.make_grid(nu_A, step, n), opts)
    for world in (3, 7):
        for r in range(world):
            k0, k1 = grid_shard(n, world, r)
            l0, l1 = halo_line_range(S["nu"], nu_A, step, k0, k1, cut)
            eng.load_lines({k: v[l0:l1] for k, v in S.items()}, assume_sorted=True)
            part = eng.cross_section(cond, xc.make_grid(nu_A + k0 * step, step, k1 - k0), opts)
            assert np.array_equal(part, full[k0:k1]), (world, r)


@pytest.mark.parametrize("profile,n_gh", [("voigt_gh_sampled", 20), ("voigt_gh_sampled", 7), ("voigt_gh_sampled", 40),
                                          ("doppler_binned", 20), ("voigt_gh_binned", 7), ("voigt_gh_binned", 40)])
@pytest.mark.parametrize("n_lines", [30, 1500])
def test_fp64_blocks_of_the_other_profiles(eng, xc, oracle_lib, profile, n_gh, n_lines):  # noqa: F811
    """FP64 blocks with other node counts (the outermost node sets the distance a block keeps) and the
    profiles without a test of their own: 1e-12, as test_fp64_blocks_against_oracle."""
    L = xs.gen_lines(317, 0, n_lines, 1000.0, 1060.0)
    E, g = xs.gen_states(317, 500)
    eng.load_lines(L)
    eng.set_states(E, g)
    n = 2049
    for nu_A, step, cut, wm, T, P in ((1010.003, 0.01, 25.0, 0.0, 900.0, 0.3), (990.0, 0.01, 25.0, 300.0, 2500.0, 10.0)):
        got = eng.cross_section(xc.make_condition(T, P), xc.make_grid(nu_A, step, n),
                                xc.make_opts(profile, "fp64", cut, wm, n_gh=n_gh))
        if profile == "voigt_gh_binned":
            Q = oracle_lib.partition_function(E, g, T)[0]
            ref = gh_binned64(L, Q, T, P, nu_A + np.arange(n) * step, step, cut, wm, n_gh)
        else:
            Q, dQ = oracle_lib.partition_function(E, g, T)
            ref = oracle_lib.cross_section(L, oracle_lib.make_condition(T, P, Q, dQ), nu_A, step, n,
                                           oracle_lib.make_opts(profile, cut, wm, n_gh), nthreads=8)
        assert metrics(got, ref)[0] < 1e-12, (profile, n_gh, nu_A)


def gh_binned64(L, Q, T, P, x, step, cut, wm, n_gh):
    """The binned Gauss-Hermite Voigt with one arctangent a node (see binned64 in test_gpu_tree)."""
    c2 = 6.62607015e-34 * 2.99792458e10 / 1.380649e-23
    nu, f = L["nu"], {k: v.astype(np.float64) for k, v in L.items()}
    al = nu * np.sqrt(2 * 1.380649e-23 * T * np.log(2) / (18 * 1.66053906660e-27)) / 2.99792458e8
    ga = f["gamma_ref"] * (296.0 / T) ** f["n_T"] * P
    S = f["g_up"] * f["A"] / (8 * np.pi * 2.99792458e10 * Q * nu ** 2) * np.exp(-c2 * f["elower"] / T)
    S = S * -np.expm1(-c2 * nu / T)
    c = np.minimum(cut, wm * np.maximum(al, ga)) if wm else np.full_like(nu, cut)
    xj, wj = np.polynomial.hermite.hermgauss(n_gh)
    out = np.empty_like(x)
    for k, xk in enumerate(x):
        D = xk - nu
        d = D[:, None] - (al / np.sqrt(np.log(2)))[:, None] * xj
        v = np.arctan2(step * ga[:, None], (d + step / 2) * (d - step / 2) + ga[:, None] ** 2) @ wj
        out[k] = (S * v)[np.abs(D) <= c].sum() * np.pi ** -1.5 / step
    return out


@pytest.mark.parametrize("n", [1, 7, 255, 2049, 32_767, 32_768, 200_001])
@pytest.mark.parametrize("nT", [1, 9])
def test_partition_function_of_many_states(xc, oracle_lib, n, nT):
    """Clusters of 8 and of 16 CTAs, shares that are empty or ragged: Q and dQ/dT to 1e-13 of the oracle
    (sums of positive terms in another order, exponentials to an ulp)."""
    E, g = xs.gen_states(318, n)
    T = np.linspace(200.0, 3000.0, nT)
    Q, dQ = xc.partition_function(E, g, T)
    for t, q, d in zip(T, Q, dQ):
        rq, rd = oracle_lib.partition_function(E, g, t)
        assert abs(q - rq) <= 1e-13 * rq and abs(d - rd) <= 1e-13 * max(abs(rd), 1e-300), (n, t)


# ------------------------------------------------------------------ sort: runs of keys that agree in their high digits
@pytest.mark.parametrize("lengths,equal", [((2, 63, 64, 65, 66, 127, 128, 129, 255, 256, 257, 1000, 2047, 2048), False),
                                           ((100, 2049), False), ((300,) * 700, False), ((65, 2048, 5000, 40_000), True),
                                           ((70_000,), True), ((66_000,), False)])
def test_sort_of_long_runs(eng, xc, lengths, equal):  # noqa: F811
    """Runs at the limits of the forms that finish them (64 keys by a thread, 2048 by a CTA, longer by every
    digit), out of order or all equal, between lines of their own: the stable order, bit for bit."""
    rng = np.random.default_rng(len(lengths) + sum(lengths))
    n = sum(lengths) + 20_000
    L = xs.gen_lines(319, 0, n, 1.0, 9000.0)
    nu, at = L["nu"], 20_000
    nu[:20_000] = np.sort(rng.uniform(1.0, 9000.0, 20_000))
    for i, m in enumerate(lengths):
        low = np.zeros(m) if equal else rng.integers(0, 2 ** 20, m) * 2.0 ** -40
        nu[at:at + m] = 2048.0 + 4.0 * i + low      # 2^-40 of 2048..8191: below the 28 leading mantissa bits
        at += m
    p = rng.permutation(n)
    L = {k: v[p] for k, v in L.items()}
    eng.load_lines(L)
    order = np.argsort(L["nu"], kind="stable")
    assert np.array_equal(eng.get_permutation(), order.astype(np.uint32))
    got = eng.get_lines()
    for k in L:
        assert np.array_equal(got[k], L[k][order]), k


def test_scratch_of_a_large_list_is_given_back(xc):
    """4e8 lines want 19 GB of scratch for one condition: it stays while calls need it, and goes when a call needs
    less than half of it or a list is loaded; the same call then gives the same bits."""
    n = 400_000_000
    with xc.Engine(0) as e:
        e.load_lines(xs.gen_lines_torch(320, 0, n, 990.0, 3010.0, device="cuda:0"))
        e.set_states(*xs.gen_states(320, 100))
        torch.cuda.synchronize()
        torch.cuda.empty_cache()

        def call(profile="voigt_w4"):
            out = e.cross_section_batched([xc.make_condition(900.0, 0.1)], xc.make_grid(2000.0, 0.01, 501),
                                          xc.make_opts(profile, "fp32", 1.0))
            return out, free - torch.cuda.mem_get_info()[0]
        free = torch.cuda.mem_get_info()[0]
        a, held = call()
        assert "block-interpolated" in e.tuning() and held > 17 << 30
        b, held = call()
        assert np.array_equal(a, b) and a.min() > 0 and held > 17 << 30
        e.set_tile_shape(8, 1)       # 16 bytes a line
        assert call()[1] < 1 << 30
        e.set_tile_shape(0, 0)
        assert np.array_equal(a, call()[0])
        e.load_lines(xs.gen_lines(320, 0, 1000, 990.0, 3010.0))
        assert free - torch.cuda.mem_get_info()[0] < 1 << 30


def test_tensor_core_far_wings_of_long_cuts(eng, xc):  # noqa: F811
    """At cuts the blocks take by themselves a fixed tile shape still runs the far wings on the tensor cores:
    against the tiled form without them and against the blocks (2e-5 as between any two FP32 paths)."""
    L = xs.gen_lines(321, 0, 30_000, 1000.0, 1100.0)
    eng.load_lines(L)
    eng.set_states(*xs.gen_states(321, 500))
    conds = [xc.make_condition(300.0 + 60.0 * i, 1e-3 * 1.33 ** i) for i in range(32)]
    grid = xc.make_grid(1000.0, 0.01, 10_001)
    blocks = eng.cross_section_batched(conds, grid, xc.make_opts("voigt_w4", "fp32", 25.0))
    assert "block-interpolated" in eng.tuning()
    eng.set_timing(True)
    eng.set_tile_shape(4, 16)
    try:
        tc = eng.cross_section_batched(conds, grid, xc.make_opts("voigt_w4", "fp32", 25.0))
        far_ms, _, _, mma = eng.sweep_kernels()
        far = eng.count_far_evals(conds, grid, xc.make_opts("voigt_w4", "fp32", 25.0))
        cores = eng.cross_section_batched(conds, grid, xc.make_opts("voigt_w4", "fp32", 25.0, tensor_cores=False))
        assert eng.sweep_kernels()[3] == 0
    finally:
        eng.set_tile_shape(0, 0)
        eng.set_timing(False)
    assert mma > 0 and far > 0 and far_ms > 0
    for ref in (cores, blocks):
        m = ref > 1e-6 * ref.max(axis=1, keepdims=True)
        assert np.max(np.abs(tc - ref)[m] / ref[m]) < 2e-5


@pytest.mark.parametrize("profile", ["voigt_w4", "lorentz", "doppler_binned", "voigt_gh_binned"])
@pytest.mark.parametrize("cut,wm", [(0.3, 0.0), (25.0, 0.0), (25.0, 300.0)])
def test_windows_inside_a_long_list(eng, xc, profile, cut, wm):  # noqa: F811
    """A narrow grid in a list that reaches far beyond it on both sides, and at either end of the list:
    constants are made for the lines in reach only (2e-5 of the general path)."""
    eng.load_lines(xs.gen_lines(322, 0, 60_000, 1000.0, 2000.0))
    eng.set_states(*xs.gen_states(322, 300))
    conds = [xc.make_condition(T, P) for T, P in ((400.0, 0.01), (1200.0, 0.5), (2600.0, 3.0))]
    for nu_A in (900.0, 974.5, 1000.0, 1500.37, 1999.0, 2030.0):
        grid, opts = xc.make_grid(nu_A, 0.01, 333), xc.make_opts(profile, "fp32", cut, wm)
        got = eng.cross_section_batched(conds, grid, opts)
        assert "block-interpolated" in eng.tuning()
        eng.set_tile_shape(8, 1)
        ref = eng.cross_section_batched(conds, grid, opts)
        eng.set_tile_shape(0, 0)
        m = ref > 1e-6 * ref.max(axis=1, keepdims=True)
        assert not m.any() or np.max(np.abs(got - ref)[m] / ref[m]) < 2e-5, nu_A


@pytest.mark.parametrize("wm", [0.0, 300.0])
@pytest.mark.parametrize("profile,n_lines,n", [("voigt_w4", 15_000, 4003), ("lorentz", 15_000, 4003),
                                               ("voigt_gh_binned", 3000, 2003), ("voigt_w4", 200, 150_003),
                                               ("doppler", 3000, 2003)])
def test_adjoint_under_a_mixture_sparse_and_dense(eng, xc, profile, n_lines, n, wm):  # noqa: F811
    """The mixture's adjoint kernels with and without blocks, fixed and width-limited cuts, 35 conditions (two
    launches): FP32 against FP64, 1e-4 of the largest."""
    eng.load_lines(xs.gen_lines(323, 0, n_lines, 2995.0, 3005.0 + 0.01 * n))
    eng.set_states(*xs.gen_states(323, 300))
    eng.set_broadening([xc.make_broadener("constant", 0.6, 0.05, 0.6), xc.make_broadener("constant", 0.4, 0.09, 0.4)])
    conds = [xc.make_condition(500.0 + 30.0 * i, 0.02 * 1.1 ** i) for i in range(35)]
    w = 1e22 * np.random.default_rng(323).uniform(0.5, 1.5, (35, n))
    grid = xc.make_grid(3000.0, 0.01, n)
    try:
        r32, r64 = (eng.cross_section_vjp_broadening(conds, grid, xc.make_opts(profile, p, 5.0, wm), w, 2)
                    for p in ("fp32", "fp64"))
    finally:
        eng.set_broadening([])
    for k in ("dT", "dP", "d_gamma_scale", "d_n_shift", "d_gamma0_broad", "d_n_broad"):
        a, b = np.asarray(r32[k]), np.asarray(r64[k])
        assert np.max(np.abs(a - b)) <= 1e-4 * max(np.max(np.abs(b)), 1e-300), k


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_gauss_hermite_adjoint_without_pressure(eng, xc, precision):  # noqa: F811
    """P = 0: no Lorentz width, and the derivatives of a bin whose edge lies exactly on a node have a pole
    (a line halfway between two grid points of a binary step, one node): finite, and the neighbours' values
    against the direct formula 1 / (s+ s-) (1e-5 FP32, 1e-12 FP64)."""
    L = xs.gen_lines(324, 0, 1, 1000.0, 1001.0)
    step, n, i0 = 1.0 / 128.0, 41, 20
    L["nu"][:] = 1000.0 + (i0 + 0.5) * step
    E, g = xs.gen_states(324, 20)
    eng.load_lines(L)
    eng.set_states(E, g)
    w = np.full((1, n), 1e22)
    cond = [xc.make_condition(296.0, 0.0)]
    r = eng.cross_section_vjp(cond, xc.make_grid(1000.0, step, n), xc.make_opts("voigt_gh_binned", precision, 25.0, n_gh=1), w)
    assert all(np.all(np.isfinite(np.asarray(v))) for v in r.values())
    sp = np.arange(n) - (i0 + 0.5) + 0.5
    sm = sp - 1.0
    ok = sp * sm != 0
    # dL/dP = I gamma_ref sum w / (h^2 pi) / (s+ s-), one node of weight sqrt(pi)
    Q = xc.partition_function(E, g, [296.0])[0][0]
    c2, f = 1.4387768775039338, {k: float(v[0]) for k, v in L.items()}
    S = f["g_up"] * f["A"] / (8 * np.pi * 2.99792458e10 * Q * f["nu"] ** 2) * np.exp(-c2 * f["elower"] / 296.0)
    S *= -np.expm1(-c2 * f["nu"] / 296.0)
    ref = S * f["gamma_ref"] * 1e22 / np.pi / step ** 2 * np.sum(1.0 / (sp * sm)[ok])
    assert abs(float(r["dP"][0]) - ref) <= (1e-5 if precision == "fp32" else 1e-12) * abs(ref)


def test_the_rule_counts_the_lines_in_reach(eng, xc):  # noqa: F811
    """A list twenty times wider than the grid is as sparse there as its part in reach; a list of the same
    length loaded afterwards over the grid alone is not."""
    grid, opts = xc.make_grid(5000.0, 0.01, 100_001), xc.make_opts("lorentz", "fp32", 25.0)
    conds = [xc.make_condition(400.0 + 60.0 * i, 0.01 * 1.3 ** i) for i in range(24)]
    eng.set_states(*xs.gen_states(325, 300))
    for lo, hi, blocks in ((0.0, 20_000.0, False), (4990.0, 6010.0, True)):
        eng.load_lines(xs.gen_lines(325, 0, 150_000, lo, hi))
        got = eng.cross_section_batched(conds, grid, opts)
        assert ("block-interpolated" in eng.tuning()) == blocks
        eng.set_tile_shape(8, 1)
        ref = eng.cross_section_batched(conds, grid, opts)
        eng.set_tile_shape(0, 0)
        m = ref > 1e-6 * ref.max(axis=1, keepdims=True)
        assert np.max(np.abs(got - ref)[m] / ref[m]) < 2e-5
