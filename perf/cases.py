"""The workloads this library's speed is judged on, each a call that a user's program makes.

A case is a line list of given size over a wavenumber range, a grid, a set of (T, P)
conditions and the options of the call.  Sizes come from the benchmark configurations in
xcsynth.WORKLOADS (the plain FP64 case, the single condition at scale, the 32-condition
sweep, differentiation and the largest list, the last three at fewer lines so that a pass
stays well below two seconds) and from the tests (a few thousand lines on a few thousand
points).

What a pass returns: a call at precision "fp64" its float64 arrays; a call at precision
"fp32" fills a float64 array with values of FP32 accuracy, which a program keeps as the
float32 opacity table (or float32 gradients) of its radiative-transfer code, so the pass
ends with that conversion.
"""
import math

import numpy as np
import torch

import paper_1801_09803_gb300 as xc
import xcsynth

DEV = "cuda:0"
MASS = 18.0
N_STATES = 5000
BASE = {
    "kind": "sweep",            # sweep | load | vjp | fit
    "profile": "voigt_w4", "precision": "fp32",
    "lines": 100_000, "lo": 1000.0, "hi": 3000.0,          # line wavenumbers, cm^-1
    "start": 1000.0, "step": 0.01, "points": 200_001,       # grid
    "cutoff": 25.0, "width_mult": 0.0,
    "nT": 1, "T0": 1000.0, "T1": 1000.0,                    # temperatures, log-spaced
    "nP": 1, "P0": 1.0, "P1": 1.0,                          # pressures, log-spaced
    "quantity": "absorption", "hitran": False, "mixture": False,
}


def case(**kw):
    c = dict(BASE)
    c.update(kw)
    return c


def listed():
    return [
        # one narrow window at one condition, called over and over (a line fit, an interactive
        # plot): latency and launches
        case(name="window_1cond", lines=2_003, lo=995.0, hi=1035.0, start=1000.0, points=3_001),
        # one absorption spectrum of a small molecule's list at one condition, FP32
        case(name="spectrum_fp32"),
        # the same in FP64, the plain form that the others are checked against
        case(name="spectrum_fp64", precision="fp64"),
        # a large list at one condition with the width-limited cut, 1 000 001 points
        case(name="width_cut_1e7", lines=10_000_000, lo=0.0, hi=10000.0, start=0.0, points=1_000_001, T0=1500.0,
             T1=1500.0, width_mult=500.0),
        # the same molecule's list thinned to its strong lines, area-conserving Gauss-Hermite Voigt
        case(name="gh_binned_5e5", profile="voigt_gh_binned", lines=500_003, lo=0.0, hi=10000.0, start=0.0,
             points=1_000_001, T0=1500.0, T1=1500.0, width_mult=500.0),
        # pressure-free (stellar) opacity: the binned Gaussian
        case(name="doppler_binned_1e6", profile="doppler_binned", lines=1_000_000, lo=0.0, hi=10000.0, start=0.0,
             points=1_000_001, T0=1500.0, T1=1500.0, width_mult=500.0),
        # the longest grid, one condition, fixed cut: a high-temperature list
        case(name="long_grid_1e7", lines=10_000_000, lo=0.0, hi=20000.0, start=0.0, points=2_000_001, T0=2000.0,
             T1=2000.0),
        # an opacity table: 8 temperatures x 4 pressures in one call
        case(name="table_32cond_1e7", lines=10_000_000, lo=0.0, hi=10000.0, start=0.0, points=1_000_001, nT=8,
             T0=300.0, T1=3000.0, nP=4, P0=1e-3, P1=10.0),
        # emission with an intensity threshold under a two-broadener mixture, an odd number of
        # conditions, a grid that covers part of the list with a ragged end
        case(name="emission_mix_7cond", lines=300_007, lo=900.0, hi=2500.0, start=1100.37, points=123_457, nT=7,
             T0=400.0, T1=2500.0, P0=0.3, P1=0.3, quantity="emission", hitran=True, mixture=True),
        # reverse mode with per-line gradients: 2 temperatures x 2 pressures
        case(name="vjp_4cond_3e5", kind="vjp", lines=300_000, nT=2, T0=800.0, T1=1600.0, nP=2, P0=0.1, P1=1.0),
        # one step of a temperature / pressure retrieval: forward, loss, backward
        case(name="fit_step_2cond", kind="fit", lines=100_000, nT=2, T0=800.0, T1=1600.0, P0=0.5, P1=0.5),
        # a fresh list: sort into wavenumber order, then the FP64 strengths and widths per line
        case(name="load_1e7", kind="load", lines=10_000_019, lo=0.0, hi=10000.0, T0=1500.0, T1=1500.0),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["sweep"] * 7 + ["vjp", "fit", "load"])
    if kind == "load":
        return case(kind=kind, lines=int(_log(rng, 1e4, 1e7)) | 1, lo=0.0, hi=10000.0, T0=round(rng.uniform(300, 3000), 1))
    step = rng.choice([0.01, 0.01, 0.02, 0.005])
    points = int(_log(rng, 3e3, 1e6 if kind == "sweep" else 2e5)) + rng.randint(0, 7)
    start = round(rng.uniform(100.0, 6000.0), 2)
    # the list covers the grid with a margin on one side and falls short of it on the other
    span = points * step
    lo, hi = max(1.0, start - rng.uniform(0.0, 30.0)), start + span * rng.uniform(0.8, 1.2) + 1.0
    c = case(kind=kind, start=start, step=step, points=points, lo=round(lo, 2), hi=round(hi, 2),
             T0=round(_log(rng, 300, 1500), 1), P0=round(_log(rng, 1e-3, 10.0), 4))
    c["T1"], c["P1"] = round(c["T0"] * rng.uniform(1.0, 2.0), 1), c["P0"]
    cap = 2e11                                             # line x point x condition evaluations
    if kind == "sweep":
        c["profile"] = rng.choice(["voigt_w4"] * 5 + ["lorentz", "doppler_binned", "voigt_gh_binned"])
        if c["profile"] == "voigt_w4" and rng.random() < 0.25:
            c["precision"], cap = "fp64", 1e9
        elif c["profile"] == "voigt_gh_binned":
            cap = 3e9
        else:
            cap = 2e10 if c["profile"] == "doppler_binned" else cap
            c["nT"], c["nP"] = rng.choice([(1, 1), (1, 1), (3, 1), (2, 2), (5, 2), (4, 4), (6, 4)])
            if c["nP"] > 1:
                c["P1"] = round(min(10.0, c["P0"] * 100.0), 4)
        if rng.random() < 0.3:
            c["width_mult"] = 500.0
        elif rng.random() < 0.3:
            c["cutoff"] = 10.0
        if c["precision"] == "fp32" and rng.random() < 0.15:
            c["quantity"], c["hitran"] = "emission", True
        if c["profile"] == "voigt_w4" and c["precision"] == "fp32" and rng.random() < 0.15:
            c["mixture"] = True
    else:
        c["nT"], c["nP"] = rng.choice([(1, 1), (2, 1), (2, 2)])
        cap = 1e10
    per_line = 2 * c["cutoff"] / step * c["nT"] * c["nP"]
    c["lines"] = int(_log(rng, 2e3, max(4e3, min(1e7, cap / per_line)))) | 1
    return c


# ---------------------------------------------------------------------------- the calls
def _temps(c):
    n = c["nT"]
    return [c["T0"] if n == 1 else c["T0"] * (c["T1"] / c["T0"]) ** (i / (n - 1)) for i in range(n)]


def _press(c):
    n = c["nP"]
    return [c["P0"] if n == 1 else c["P0"] * (c["P1"] / c["P0"]) ** (i / (n - 1)) for i in range(n)]


def _tp(c):
    return [(T, P) for T in _temps(c) for P in _press(c)]


def _threshold(c):
    # HITRAN's dynamic cut; emissivities are in erg/s/sr per molecule
    if not c["hitran"]:
        return None
    return ("hitran", 2000.0, 1e-29 if c["quantity"] == "absorption" else 1e-22)


_TABLE = {J: (0.05 + 0.04 / (1 + 0.1 * J), 0.75 - 0.004 * J) for J in range(0, 41)}   # gamma_0, n by J''


def _broadeners():
    return [xc.make_broadener("a0", 0.85, 0.06, 0.55, _TABLE), xc.make_broadener("constant", 0.15, 0.04, 0.5)]


def _lines(c, seed):
    return xcsynth.gen_lines_torch(180109803 + 1000 * seed, 0, c["lines"], c["lo"], c["hi"], device=DEV)


def prepare(case, seed):
    c = case
    s = {"case": c}
    lines = _lines(c, seed)
    E, g = xcsynth.gen_states(180109803 + seed, N_STATES)
    eng = xc.Engine(0)
    eng.set_states(E, g)
    s["eng"] = eng
    s["conds"] = [xc.make_condition(T, P, mass_da=MASS) for T, P in _tp(c)]
    if c["kind"] == "load":
        s["lines"] = lines
        s["params"] = [torch.empty(c["lines"], dtype=torch.float64, device=DEV) for _ in range(3)]
        return s
    eng.load_lines(lines)
    if c["mixture"]:
        eng.set_broadening(_broadeners())
    s["grid"] = xc.make_grid(c["start"], c["step"], c["points"])
    s["opts"] = xc.make_opts(c["profile"], c["precision"], c["cutoff"], c["width_mult"], quantity=c["quantity"],
                             threshold=_threshold(c))
    shape = (len(s["conds"]), c["points"])
    if c["kind"] == "sweep":
        s["out"] = torch.empty(shape, dtype=torch.float64, device=DEV)
    else:
        s["w"] = _weights(c, seed)
        if c["kind"] == "fit":
            tp = torch.tensor(_tp(c), dtype=torch.float64)
            s["T"] = tp[:, 0].clone().requires_grad_(True)
            s["P"] = tp[:, 1].clone().requires_grad_(True)
            s["scale"] = torch.tensor(1.0, dtype=torch.float64, requires_grad=True)
            s["shift"] = torch.tensor(0.0, dtype=torch.float64, requires_grad=True)
    return s


def _weights(c, seed):
    """dL/dsigma of a weighted fit: noise-like weights of the size of 1 / sigma."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    return 1e22 * torch.rand((c["nT"] * c["nP"], c["points"]), dtype=torch.float64, device=DEV, generator=gen)


def run(state):
    c, eng = state["case"], state["eng"]
    if c["kind"] == "load":
        eng.load_lines(state["lines"])
        eng.line_params_device(state["conds"][0], *state["params"])
        return state["params"]
    if c["kind"] == "sweep":
        eng.cross_section_batched(state["conds"], state["grid"], state["opts"], state["out"])
        return state["out"] if c["precision"] == "fp64" else state["out"].float()
    if c["kind"] == "vjp":
        r = eng.cross_section_vjp(state["conds"], state["grid"], state["opts"], state["w"])
        return {k: v.float() for k, v in r.items()}
    par = [state[k] for k in ("T", "P", "scale", "shift")]
    for p in par:
        p.grad = None
    sigma = xc.cross_section_autograd(eng, *par, state["grid"], state["opts"], mass_da=MASS)
    (state["w"] * sigma).sum().backward()
    return [sigma.detach().float()] + [p.grad.float() for p in par]


def _evals(c):
    """Line x point x condition evaluations inside the fixed cut, for lines spread evenly over
    (lo, hi] (the width-limited cut: the widths of a line in the middle of the list)."""
    cut = c["cutoff"]
    if c["width_mult"]:
        nu = 0.5 * (c["lo"] + c["hi"])
        T = c["T0"]
        w = max(3.581e-7 * nu * math.sqrt(T / MASS), 0.06 * (296.0 / T) ** 0.6 * c["P0"])
        cut = min(cut, c["width_mult"] * w)
    a, b = c["start"], c["start"] + (c["points"] - 1) * c["step"]
    x = np.linspace(c["lo"], c["hi"], 4001)
    cover = np.maximum(0.0, np.minimum(b, x + cut) - np.maximum(a, x - cut)).mean() / c["step"]
    return c["lines"] * cover * c["nT"] * c["nP"]


def work(case):
    """Bytes: the 28-byte line records and the outputs, once each (a load also writes the sorted
    records; the adjoint reads dL/dsigma).  Flops: 10 per line x point x condition of the sum
    as the method states it (one region-I Voigt evaluation); a load computes per line only."""
    c = case
    n, out = c["lines"], 8 * c["points"] * c["nT"] * c["nP"]
    if c["kind"] == "load":
        return {"bytes": n * (28 + 28 + 28 + 24), "flops": 60 * n}
    ev = _evals(c)
    per = {"voigt_gh_binned": 200, "doppler_binned": 20, "lorentz": 5}.get(c["profile"], 10)
    if c["kind"] == "sweep":
        return {"bytes": 28 * n + out, "flops": per * ev}
    if c["kind"] == "vjp":
        return {"bytes": 28 * n + out + 16 * n, "flops": 3 * per * ev}
    return {"bytes": 2 * 28 * n + 3 * out, "flops": 4 * per * ev}


# ---------------------------------------------------------------------------- in 64 bits
H_, C_, K_, DA_ = 6.62607015e-34, 2.99792458e8, 1.380649e-23, 1.66053906660e-27
C2_ = H_ * C_ * 100.0 / K_
LN2 = math.log(2.0)
_SKIP = 3e10        # line x point x condition evaluations that stay within some seconds


def _w4(x, y):
    """Re w(x + iy), x >= 0, by Humlicek's w4 (JQSRT 27, 437) for |x| + y < 15."""
    t = torch.complex(y, -x)
    s = x + y
    u = t * t
    r2 = (t * (1.410474 + u * 0.5641896) / (0.75 + u * (3.0 + u))).real
    n3 = 16.4955 + t * (20.20933 + t * (11.96482 + t * (3.778987 + t * 0.5642236)))
    d3 = 16.4955 + t * (38.82363 + t * (39.27121 + t * (21.69274 + t * (6.699398 + t))))
    r3 = (n3 / d3).real
    n4 = 36183.31 - u * (3321.9905 - u * (1540.787 - u * (219.0313 - u * (35.76683 - u * (1.320522 - u * 0.56419)))))
    d4 = 32066.6 - u * (24322.84 - u * (9022.228 - u * (2186.181 - u * (364.2191 - u * (61.57037 - u * (1.841439 - u))))))
    four = (s < 5.5) & (y < 0.195 * x - 0.176)
    # no overflow of exp where region IV is not used
    ue = torch.where(four, u, torch.zeros_like(u))
    r4 = (torch.exp(ue) - t * n4 / d4).real
    return torch.where(s >= 5.5, r2, torch.where(four, r4, r3))


def _voigt(D, al, ga):
    """Unit-area Voigt by w4 at offsets D[l, k] of lines with widths al[l], ga[l]."""
    ia = (math.sqrt(LN2) / al)[:, None]
    x, y = D.abs() * ia, (ga[:, None] * ia)
    X, Y = x * x, y * y
    t = X + Y - 0.5
    w = 0.5641896 * y * (0.5 + X + Y) / (t * t + 2.0 * Y)
    i = torch.nonzero((x + y < 15.0).reshape(-1)).reshape(-1)
    if i.numel():
        yy = y.expand_as(x).reshape(-1)[i]
        w = w.reshape(-1).index_put((i,), _w4(x.reshape(-1)[i], yy)).reshape(x.shape)
    return w * (math.sqrt(LN2 / math.pi) / al)[:, None]


def _profile(c, D, al, ga, nodes):
    h = c["step"]
    if c["profile"] == "voigt_w4":
        return _voigt(D, al, ga)
    if c["profile"] == "lorentz":
        g = ga[:, None]
        return g / (math.pi * (D * D + g * g))
    if c["profile"] == "doppler_binned":
        k, t = (math.sqrt(LN2) / al)[:, None], D.abs()
        return (torch.special.erfc(k * (t - 0.5 * h)) - torch.special.erfc(k * (t + 0.5 * h))) / (2.0 * h)
    g, v = ga[:, None], 0.0
    for xj, wj in zip(*nodes):
        d = D - (al * (xj / math.sqrt(LN2)))[:, None]
        v = v + wj * torch.atan2(h * g, (d + 0.5 * h) * (d - 0.5 * h) + g * g)
    return v * (math.pi ** -1.5 / h)


def _params(c, L, T, P, scale, shift, E, g, gref=None, nT=None):
    """Strength, Doppler and Lorentz half-widths per line (float64)."""
    nu, el, A, gu = L["nu"], L["elower"].double(), L["A"].double(), L["g_up"].double()
    Q = (g * torch.exp(-C2_ * E / T)).sum()
    if c["quantity"] == "emission":
        S = gu * A * (H_ * 1e7 * C_ * 100.0) * nu / (4.0 * math.pi) * torch.exp(-C2_ * (el + nu) / T) / Q
    else:
        S = gu * A / (8.0 * math.pi * C_ * 100.0 * nu * nu) * torch.exp(-C2_ * el / T) * -torch.expm1(-C2_ * nu / T) / Q
    if c["hitran"]:
        _, nc, ic = _threshold(c)
        S = torch.where(S < torch.where(nu > nc, torch.full_like(nu, ic), ic * nu / nc * torch.tanh(C2_ * nu / T / 2)),
                        torch.zeros_like(S), S)
    al = nu * torch.sqrt(2.0 * K_ * LN2 * T / (MASS * DA_)) / C_
    if c["mixture"]:
        jl = L["j_lo"].long()
        tg = torch.tensor([_TABLE[j][0] if j in _TABLE else 0.06 for j in range(128)], dtype=torch.float64, device=DEV)
        tn = torch.tensor([_TABLE[j][1] if j in _TABLE else 0.55 for j in range(128)], dtype=torch.float64, device=DEV)
        ga = P * scale * (0.85 * tg[jl] * (296.0 / T) ** (tn[jl] + shift) + 0.15 * 0.04 * (296.0 / T) ** (0.5 + shift))
    else:
        ga = scale * gref * (296.0 / T) ** (nT + shift) * P
    return S, al, ga


def exact(case, seed):
    c = case
    if c["kind"] != "load" and _evals(c) * {"voigt_gh_binned": 10}.get(c["profile"], 1) \
            * (1 if c["kind"] == "sweep" else 3) > _SKIP * (1 if c["kind"] == "sweep" else 0.8):
        return None
    L = _lines(c, seed)
    order = torch.argsort(L["nu"], stable=True)
    L = {k: v[order] for k, v in L.items()}
    E, g = xcsynth.gen_states(180109803 + seed, N_STATES)
    E, g = torch.tensor(E, device=DEV), torch.tensor(g, device=DEV).double()
    tp = torch.tensor(_tp(c), dtype=torch.float64, device=DEV)
    diff = c["kind"] in ("vjp", "fit")
    leaf = lambda v: v.detach().clone().requires_grad_(diff)  # noqa: E731
    T, P, scale, shift = leaf(tp[:, 0]), leaf(tp[:, 1]), leaf(tp.new_tensor(1.0)), leaf(tp.new_tensor(0.0))
    gref, nT = leaf(L["gamma_ref"].double()), leaf(L["n_T"].double())
    if c["kind"] == "load":
        return list(_params(c, L, T[0], P[0], scale, shift, E, g, gref, nT))
    x, w = np.polynomial.hermite.hermgauss(20)
    nodes = (x.tolist(), w.tolist())
    out = torch.zeros((tp.shape[0], c["points"]), dtype=torch.float64, device=DEV)
    wts = _weights(c, seed) if diff else None
    nu, h = L["nu"], c["step"]
    density = c["lines"] / max(c["hi"] - c["lo"], 1e-9)
    W = 256
    while W < 4096 and W * (2 * c["cutoff"] + W * h) * density < 4e6:
        W *= 2
    starts = list(range(0, c["points"], W))
    xs0 = torch.tensor([c["start"] + k * h for k in starts], dtype=torch.float64, device=DEV)
    xs1 = torch.tensor([c["start"] + (min(k + W, c["points"]) - 1) * h for k in starts], dtype=torch.float64, device=DEV)
    a = torch.searchsorted(nu, xs0 - c["cutoff"] * (1 + 1e-9) - 1e-6).tolist()
    b = torch.searchsorted(nu, xs1 + c["cutoff"] * (1 + 1e-9) + 1e-6, right=True).tolist()
    for ci in range(tp.shape[0]):
        S, al, ga = _params(c, L, T[ci], P[ci], scale, shift, E, g, gref, nT)
        Sd, ad, gd = (v.detach().requires_grad_(diff) for v in (S, al, ga))
        cut = torch.full_like(nu, c["cutoff"])
        if c["width_mult"]:
            cut = torch.minimum(cut, c["width_mult"] * torch.maximum(ad, gd)).detach()
        acc = [torch.zeros_like(nu) for _ in range(3)] if diff else None
        for k0, i0, i1 in zip(starts, a, b):
            k1 = min(k0 + W, c["points"])
            xk = c["start"] + torch.arange(k0, k1, dtype=torch.float64, device=DEV) * h
            m = max(1, int(1.5e7 if diff else 3e7) // (k1 - k0))
            for j0 in range(i0, i1, m):
                j = slice(j0, min(j0 + m, i1))
                p = [v[j].detach().requires_grad_(diff) for v in (Sd, ad, gd)]
                D = xk[None, :] - nu[j, None]
                V = torch.where(D.abs() <= cut[j, None], _profile(c, D, p[1], p[2], nodes), torch.zeros((), dtype=torch.float64, device=DEV))
                sig = p[0] @ V
                out[ci, k0:k1] += sig.detach()
                if diff:
                    for q, v in zip(acc, torch.autograd.grad((wts[ci, k0:k1] * sig).sum(), p)):
                        q[j] += v
        if diff:
            torch.autograd.backward([S, al, ga], acc)
    if not diff:
        return out
    one = lambda v: v.grad.reshape(-1)  # noqa: E731
    if c["kind"] == "vjp":
        return {"dT": one(T), "dP": one(P), "d_gamma_scale": one(scale), "d_n_shift": one(shift),
                "d_gamma_ref_line": one(gref), "d_n_line": one(nT)}
    return [out, one(T), one(P), scale.grad, shift.grad]
