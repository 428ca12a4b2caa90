"""The rule of the block-interpolated FP32 sweep (csrc/xc_tree.cu), emulated on the CPU.

Every (line, grid point) pair inside the cut must be counted exactly once, by the largest
block that takes the line or at the point itself, and the candidate ranges that a block
scans must hold every line it takes -- for fixed and per-line cuts, ragged grids, lines off
the grid and cuts shorter than a block.  And the interpolation error of a block's 16
(rounded) nodes for the nearest line it takes stays below FP32 rounding of the profile."""
import numpy as np
import pytest

BLOCK = (64, 128, 512)
GAP = (36, 72, 284)


def node(B, m):
    return np.round(64.0 * (B - 1) * (1.0 - np.cos(np.pi * (2 * m + 1) / 32.0))) / 128.0


def radius(lev, b1, per_step, reach, ext, ext0, core):
    """tr_radius: the same for every line, growing with level and position."""
    ah = per_step * max(b1 + reach, 0)
    return max(GAP[lev] + ext0 + int(np.ceil(ah * ext)), int(np.ceil(ah * core)) + 2)


def takes(n, ka, kb, b0, b1, N, D):
    return (ka <= b0) & (kb >= min(b1, N - 1)) & ((n < b0 - D) | (n > b1 + D))


def far_ranges(b0, b1, N, D, reach, cover, parent):
    a, z = min(b1, N - 1) - reach, b0 - D
    a2, z2 = b1 + D + 1, b0 + reach + 1
    e1, s2, e3, s4 = z, z, z2, z2
    if parent:
        p0, p1, Dp = parent
        e1 = min(z, max(a, p1 - cover))
        s2 = min(z, max(e1, p0 - Dp))
        e3 = min(z2, p1 + Dp + 1)
        s4 = min(z2, max(e3, p0 + cover))
    return [(a, e1), (s2, z), (a2, e3), (s4, z2)]


def point_ranges(s0, s1, p0, p1, Dp, reach, cover):
    a, z = s0 - reach, s1 + reach + 1
    e1 = max(a, min(p0 - Dp, p1 - cover))
    s2 = max(e1, p0 - Dp)
    e2 = min(z, p1 + Dp + 1)
    return [(a, e1), (s2, e2), (min(z, max(e2, p0 + cover)), z)]


@pytest.mark.parametrize("N", [1, 31, 33, 64, 65, 500, 513, 1537])
@pytest.mark.parametrize("cut,per_line", [(2500, False), (700, False), (90, False), (900, True), (20, True)])
@pytest.mark.parametrize("per_step,core", [(0.0, 0.0), (2e-4, 18.05), (4e-3, 18.05)])
def test_every_pair_once(N, cut, per_line, per_step, core):
    rng = np.random.default_rng(N * 7 + cut)
    pos = np.sort(np.concatenate([rng.uniform(-cut - 40, N + cut + 40, 300), rng.uniform(-5, N + 5, 60)]))
    n = np.floor(pos).astype(int)
    c = rng.uniform(0.02, 1.0, len(pos)) * cut if per_line else np.full(len(pos), float(cut))
    ka = np.maximum(np.ceil(pos - c).astype(int), 0)
    kb = np.minimum(np.floor(pos + c).astype(int), N - 1)
    ka, kb = np.where(kb < ka, 1, ka), np.where(kb < ka, 0, kb)
    reach, cover = cut + 2, 0 if per_line else max(0, cut - 2)
    # alpha in grid steps: per_step times the position, as alpha = (alpha / nu) nu
    rad = lambda lev, b1: radius(lev, b1, per_step, reach, 0.86, 2, core)  # noqa: E731
    count = np.zeros((len(pos), N), int)
    taken = {}
    for lev in (2, 1, 0):
        B = BLOCK[lev]
        for b0 in range(0, N, B):
            b1, D = b0 + B - 1, rad(lev, b0 + B - 1)
            own = takes(n, ka, kb, b0, b1, N, D)
            parent = None
            if lev < 2:
                P = BLOCK[lev + 1]
                p0 = b0 // P * P
                parent = (p0, p0 + P - 1, rad(lev + 1, p0 + P - 1))
                up = taken[lev + 1, p0]
                assert not np.any(up & ~own)          # a child takes what its parent takes
                own_new = own & ~up
            else:
                own_new = own
            taken[lev, b0] = own
            cand = np.zeros(len(pos), int)
            for a, z in far_ranges(b0, b1, N, D, reach, cover, parent):
                cand += (n >= a) & (n < z)
            assert np.all(cand <= 1) and np.all(cand[own_new] == 1)
            k1 = min(b1, N - 1)
            assert np.all(ka[own_new] <= b0) and np.all(kb[own_new] >= k1)
            count[own_new, b0:k1 + 1] += 1
    for s0 in range(0, N, 32):
        s1, p0 = s0 + 31, s0 // 64 * 64
        Dp = rad(0, p0 + 63)
        ok = (ka <= s1) & (kb >= s0) & (ka <= kb) & ~taken[0, p0]
        cand = np.zeros(len(pos), int)
        for a, z in point_ranges(s0, s1, p0, p0 + 63, Dp, reach, cover):
            cand += (n >= a) & (n < z)
        assert np.all(cand <= 1) and np.all(cand[ok] == 1)
        for k in range(s0, min(s1, N - 1) + 1):
            count[:, k] += ok & (ka <= k) & (k <= kb)
    k = np.arange(N)
    assert np.array_equal(count, ((k[None] >= ka[:, None]) & (k[None] <= kb[:, None])).astype(int))


@pytest.mark.parametrize("B,gap", list(zip(BLOCK, GAP)))
def test_interpolation_error_of_the_nearest_line(B, gap):
    """1/(x - s)^2 with s on the real axis `gap` steps from the block (other pole positions are
    farther from it): the bound stated in the source, 2e-8 of every value."""
    xn = node(B, np.arange(16))
    x = np.arange(B, dtype=float)
    L = np.array([np.prod([(x - xn[j]) / (xn[m] - xn[j]) for j in range(16) if j != m], axis=0) for m in range(16)])
    assert np.abs(L).sum(0).max() < 3.0
    for s in (-float(gap), B - 1.0 + gap):
        f = lambda t: 1.0 / (t - s) ** 2  # noqa: E731
        assert np.max(np.abs(f(xn) @ L - f(x)) / f(x)) < 2e-8
