"""The work a user of this framework has it do, as measurable cases.

Each case goes through the public entry points of ``paper_1502_07873_gb300`` the way the
README, the benchmark and the server use them: a context on a grid, the autotuner once,
then forward solves, Gauss-Newton Hessians, gains, design sweeps, Newton estimates or
double-loop Monte Carlo.  Grids, media, receivers, priors and node counts are those of the
repository's workloads (2 km x 1 km half-plane, the paper's LOH.1-like box) or lie between
them.

``exact`` restates the method in plain torch in 64 bits: the regularised source, the
leap-frog scheme with its free surface and absorbing rows, Jacobians, Hessians, gains.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1502_07873_gb300 as P

DEV = "cuda"

# (z_top, vp, vs, rho) per layer
MEDIA = {
    "homogeneous": ((0.0, 3000.0, 1732.0, 2500.0),),
    "three_layer": ((0.0, 2000.0, 1155.0, 2200.0), (300.0, 3000.0, 1732.0, 2500.0), (600.0, 4500.0, 2598.0, 2700.0)),
    "paper": ((0.0, 4000.0, 2000.0, 2600.0), (1000.0, 6000.0, 3464.0, 2700.0)),
}
# prior boxes of (x_s, z_s, t_s, omega_s, m_xx, m_xz, m_zz)
PRIORS = {
    "half_plane": ((800.0, 400.0, 0.1, 4.0, 1e13, 1e13, 1e13), (1200.0, 600.0, 0.3, 8.0, 1e14, 1e14, 1e14)),
    "paper": ((9000.0, 1000.0, 0.5, 3.0, 1e13, 1e13, 1e13), (11000.0, 3000.0, 1.5, 5.0, 1e15, 1e15, 1e15)),
}
PAPER_KNOWN = (9000.0, 2000.0, 1.0, 4.0, 1e14, 1e14, 1e14)   # the paper's three-unknown studies
PAPER_UNKNOWN = (1, 3, 4)                                    # depth, omega_s, m_xx
REL_STEP = 1e-4
JACOBIANS = {"pairs": 0, "difference": 1, "sensitivity": 2}
MAX_CHUNK = 2048   # nodes per chunk of a context, as the paper's scenarios run


def _half_plane(nx, medium, seconds, nrec):
    """Grid fields of a 2 km wide, about 1 km deep half-plane at CFL 0.5."""
    h = 2000.0 / (nx - 1)
    dt = 0.5 * h / max(l[1] for l in MEDIA[medium])
    return {"nx": nx, "nz": int(round(1000.0 / h)) + 1, "h": h, "dt": dt, "nsteps": int(math.ceil(seconds / dt - 1e-9)),
            "medium": medium, "nrec": nrec, "prior": "half_plane"}


def _paper_box(nsteps, nrec):
    """The paper's model problem: 20 km x 15 km at h = 200 m, dt = 0.025 s."""
    return {"nx": 101, "nz": 76, "h": 200.0, "dt": 0.025, "nsteps": nsteps, "medium": "paper", "nrec": nrec,
            "prior": "paper"}


def listed():
    hp, pb = _half_plane, _paper_box
    return [
        # one source, one answer: a user trying a source by hand; latency and launches count
        dict(hp(81, "homogeneous", 1.6666, 5), name="forward_81x41_one_source", kind="forward", n=1, fp64=False),
        # the small parity workload: 16 Monte Carlo nodes, everything in FP64
        dict(hp(81, "homogeneous", 1.6666, 5), name="eig_81x41_fp64_pairs", kind="eig", n=16, fp64=True,
             jac="pairs", sigma=0.05),
        # the benchmark: a whole EIG evaluation from host buffers, 256 nodes, 3840 solves
        dict(hp(401, "homogeneous", 1.6666, 20), name="eig_host_401x201_pairs", kind="host", n=256, fp64=False,
             jac="pairs", sigma=0.29),
        # part of the layered workload: a grid too large for the chip, 4000 steps
        dict(hp(801, "three_layer", 1.1111, 40), name="eig_801x401_layered", kind="eig", n=8, fp64=False,
             jac="difference", sigma=0.29),
        # the serving mix's largest grid: few solves, each of them large
        dict(hp(1601, "three_layer", 0.5, 23), name="eig_1601x801_layered", kind="eig", n=1, fp64=False,
             jac="difference", sigma=0.29),
        # the serving mix's smallest grid
        dict(hp(201, "three_layer", 0.5, 17), name="eig_201x101_layered", kind="eig", n=64, fp64=False,
             jac="difference", sigma=0.29),
        # design sweep, first half: partial Hessians per receiver and time window
        dict(hp(401, "homogeneous", 2.0, 40), name="windows_401x201", kind="windows", n=32, fp64=False,
             jac="difference", sigma=0.29, windows="0.5 1.0 2.0"),
        # design sweep, second half: the gain of every candidate receiver subset in one window
        {"name": "designs_5120_of_40", "kind": "designs", "n": 1024, "nrec": 40, "nwin": 3, "win": 1, "per_k": 512},
        # the paper's scenarios: 91 candidate receivers, sensitivity solves, 36 line designs
        dict(pb(320, 91), name="scenarios_101x76", kind="scenarios", n=1024, fp64=False, jac="sensitivity", sigma=0.01),
        # the paper's convergence study: short records at two receivers, many nodes, three unknowns
        dict(pb(50, 2), name="study_101x76_subset", kind="study", n=8583, fp64=False, jac="sensitivity", sigma=0.01),
        # the refined gain: Newton iterations with the dual solve, everything in FP64
        dict(pb(50, 2), name="newton_101x76_fp64", kind="map", n=256, fp64=True, jac="sensitivity", sigma=0.01, iters=2),
        # the nested Monte Carlo estimate the Laplace form is checked against
        dict(pb(50, 2), name="double_loop_4096", kind="dlmc", n=4096, m=4096, sigma=0.01),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(("forward", "eig", "eig", "eig", "host", "windows", "designs", "scenarios", "study", "map", "dlmc"))
    if kind == "designs":
        nwin = rng.randint(1, 3)
        return {"kind": kind, "n": _log(rng, 33, 1500), "nrec": rng.randint(11, 91), "nwin": nwin,
                "win": rng.randrange(nwin), "per_k": _log(rng, 5, 600)}
    if kind == "dlmc":
        return dict(_paper_box(rng.randint(17, 70), 2), kind=kind, n=_log(rng, 65, 5000), m=_log(rng, 65, 5000), sigma=0.01)
    if kind == "map":
        return dict(_paper_box(rng.randint(30, 80), rng.randint(2, 9)), kind=kind, n=_log(rng, 5, 400), fp64=True,
                    jac="sensitivity", sigma=0.01, iters=rng.randint(0, 3))
    if kind == "study":
        return dict(_paper_box(rng.randint(30, 80), rng.randint(1, 9)), kind=kind, n=_log(rng, 33, 9000), fp64=False,
                    jac="sensitivity", sigma=0.01)
    if kind == "scenarios":
        return dict(_paper_box(rng.randint(100, 320), 91), kind=kind, n=_log(rng, 15, 1100), fp64=False,
                    jac="sensitivity", sigma=0.01)
    nx = _log(rng, 61, 1601)
    fp64 = kind != "windows" and nx < 300 and rng.random() < 0.25
    c = _half_plane(nx, rng.choice(("homogeneous", "three_layer")), rng.uniform(0.5, 0.9), rng.randint(5, 40))
    per = 1
    c.update(kind=kind, fp64=fp64)
    if kind != "forward":
        c.update(jac="difference" if kind == "windows" else rng.choice(("pairs", "difference", "sensitivity")), sigma=0.29)
        per = 15 if c["jac"] == "pairs" else 7
    if kind == "windows":
        c["windows"] = "0.45 0.5"
    top = (3e9 if fp64 else 4e10) / (c["nx"] * c["nz"] * c["nsteps"] * per)
    c["n"] = _log(rng, 1, max(1.0, min(256.0, top)))
    return c


# ------------------------------------------------------------------------- inputs

def _receivers(case):
    if case["prior"] == "paper":   # the candidates of the scenarios, or positions spread over the same line
        if case["nrec"] == 91:
            return list(range(5, 96))
        return [5 + int(round(50.0 * (r + 1) / case["nrec"])) if r else 5 for r in range(case["nrec"])]
    lx = (case["nx"] - 1) * case["h"]
    return [int(math.floor((r + 0.5) * lx / case["nrec"] / case["h"] + 0.5)) for r in range(case["nrec"])]


def _thetas(case, n, seed):
    rng = np.random.default_rng(seed)
    lo, hi = (np.array(v) for v in PRIORS[case["prior"]])
    if case["kind"] in ("study", "map", "dlmc"):
        th = np.tile(np.array(PAPER_KNOWN), (n, 1))
        for j in PAPER_UNKNOWN:
            th[:, j] = lo[j] + (hi[j] - lo[j]) * rng.random(n)
        return th
    return lo + (hi - lo) * rng.random((n, 7))


def _win_levels(case):
    if case["kind"] == "scenarios":
        return [case["nsteps"] + 1]
    return [min(case["nsteps"] + 1, int(math.floor(t / case["dt"] + 1e-9)) + 1) for t in map(float, case["windows"].split())]


def _noise(case, shape, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    return case["sigma"] * torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen)


def _line_designs():
    """The paper's 36 designs as masks over the 91 candidates (200 m apart): more receivers
    over a fixed span, more receivers at a fixed spacing, five receivers at growing spacings."""
    rows = []
    for n, d in [(3, 40), (5, 20), (9, 10), (17, 5), (41, 2), (81, 1)] + [(n, 5) for n in range(1, 20, 2)] + \
            [(5, d) for d in range(1, 21)]:
        m = np.zeros(91, dtype=np.uint8)
        m[[45 + (2 * k - (n - 1)) * d // 2 for k in range(n)]] = 1
        rows.append(m)
    return np.stack(rows)


def _subset_designs(case, seed):
    """Random receiver subsets: per_k of every size 1..10."""
    rng = np.random.default_rng(seed)
    rows = np.zeros((10 * case["per_k"], case["nrec"]), dtype=np.uint8)
    for i in range(rows.shape[0]):
        rows[i, rng.choice(case["nrec"], size=1 + i // case["per_k"], replace=False)] = 1
    return rows


def _partial_hessians(case, seed):
    """Per-receiver, per-window partial Hessians, as sums of J^T J over growing windows, with
    the parameters' own scales and correlated columns."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    lo, hi = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in PRIORS["half_plane"])
    n, nrec, nwin = case["n"], case["nrec"], case["nwin"]
    iu = torch.triu_indices(7, 7, device=DEV)
    out = torch.empty((n, nrec, nwin, 28), dtype=torch.float64, device=DEV)
    H = torch.zeros((n, nrec, 7, 7), dtype=torch.float64, device=DEV)
    for k in range(nwin):
        J = torch.randn((n, nrec, 24, 7), dtype=torch.float64, device=DEV, generator=gen)
        J = (J + 0.5 * J.roll(1, -1)) * (40.0 / (hi - lo))
        H += J.transpose(-1, -2) @ J
        out[:, :, k] = H[..., iu[0], iu[1]]
    return out


def prepare(case, seed):
    kind = case["kind"]
    lo, hi = PRIORS[case.get("prior", "half_plane")]
    st = {"kind": kind, "lo": lo, "hi": hi, "case": case}
    if kind == "designs":
        st["H_rec"] = _partial_hessians(case, seed)
        st["mask"] = torch.tensor(_subset_designs(case, seed), device=DEV)
        st["w"] = torch.full((case["n"],), 1.0 / case["n"], dtype=torch.float64, device=DEV)
        nd = st["mask"].shape[0]
        st["eig"] = torch.empty(nd, dtype=torch.float64, device=DEV)
        st["n_bad"] = torch.empty(nd, dtype=torch.int32, device=DEV)
        return st
    if kind == "dlmc":   # seismograms of the outer and the inner samples, and the noise
        n, m = case["n"], case["m"]
        g = _seismograms(case, np.concatenate([_thetas(case, n, seed), _thetas(case, m, seed + 7919)])).flatten(1)
        st["g_out"], st["g_in"] = g[:n].contiguous(), g[n:].contiguous()
        st["eps"] = _noise(case, tuple(st["g_out"].shape), seed)
        st["log_ev"] = torch.empty(n, dtype=torch.float64, device=DEV)
        st["eig"] = torch.empty(1, dtype=torch.float64, device=DEV)
        return st
    n = case["n"]
    prob = P.make_problem(case["nx"], case["nz"], case["h"], case["dt"], case["nsteps"], MEDIA[case["medium"]],
                          _receivers(case), P.OED_FP64 if case["fp64"] else P.OED_FP32)
    per = 1 if kind == "forward" else (15 if case["jac"] == "pairs" else 7)
    ctx = P.Context(prob, max_solves=max(per, min(n, MAX_CHUNK) * per))
    if kind != "forward":
        ctx.jacobian = JACOBIANS[case["jac"]]
    ctx.autotune(min(n, MAX_CHUNK) * per)
    th = _thetas(case, n, seed)
    st["ctx"] = ctx
    if kind == "host":
        st["theta"] = torch.tensor(th).pin_memory()
        st["w"] = torch.full((n,), 1.0 / n, dtype=torch.float64).pin_memory()
        return st
    st["theta"] = torch.tensor(th, device=DEV)
    if kind == "forward":
        st["g"] = torch.empty((n, ctx.nlev, ctx.nrec, 2), dtype=torch.float64, device=DEV)
        return st
    st["w"] = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    st["H"] = torch.empty((n, 7, 7), dtype=torch.float64, device=DEV)
    st["status"] = torch.empty(n, dtype=torch.int32, device=DEV)
    if kind == "map":
        y = _seismograms(case, _thetas(case, n, seed))
        st["y"] = (y + _noise(case, tuple(y.shape), seed)).contiguous()
        st["grad"] = torch.empty((n, 7), dtype=torch.float64, device=DEV)
        return st
    if kind in ("windows", "scenarios"):
        st["wl"] = _win_levels(case)
        st["H_rec"] = torch.empty((n, ctx.nrec, len(st["wl"]), 28), dtype=torch.float64, device=DEV)
    nd = 1
    if kind == "scenarios":
        st["mask"] = torch.tensor(_line_designs(), device=DEV)
        nd = st["mask"].shape[0]
    st["eig"] = torch.empty(nd, dtype=torch.float64, device=DEV)
    st["n_bad"] = torch.empty(nd, dtype=torch.int32, device=DEV)
    st["dkl"] = torch.empty(n, dtype=torch.float64, device=DEV)
    return st


# --------------------------------------------------------------------------- one pass

def run(st):
    kind, c, lo, hi = st["kind"], st["case"], st["lo"], st["hi"]
    if kind == "designs":
        P.oed_eig_designs(None, st["H_rec"], c["win"], st["mask"], st["w"], lo, hi, st["eig"], n_bad=st["n_bad"])
        return {"eig": st["eig"], "n_bad": st["n_bad"]}
    if kind == "dlmc":
        P.oed_dlmc(st["g_out"], st["eps"], st["g_in"], c["sigma"], st["log_ev"], st["eig"])
        return {"log_ev": st["log_ev"], "eig": st["eig"]}
    if kind == "forward":
        P.oed_forward(st["ctx"], st["theta"], st["g"])
        return {"g": st["g"]}
    if kind == "host":
        eig, dkl, bad = P.oed_eig_host(st["ctx"], st["theta"], st["w"], lo, hi, REL_STEP, c["sigma"], want_dkl=True)
        return {"eig": eig, "dkl": dkl, "n_bad": bad}
    if kind == "map":
        theta = st["theta"].clone()
        P.oed_hessian_map(st["ctx"], theta, st["y"], lo, hi, REL_STEP, c["sigma"], c["iters"], st["H"], st["grad"],
                          free=PAPER_UNKNOWN, status=st["status"])
        return {"theta": theta, "H": st["H"], "grad": st["grad"], "status": st["status"]}
    P.oed_hessian(st["ctx"], st["theta"], lo, hi, REL_STEP, c["sigma"], st["H"], win_levels=st.get("wl"),
                  H_rec=st.get("H_rec"), status=st["status"])
    out = {"H": st["H"], "status": st["status"], "eig": st["eig"], "n_bad": st["n_bad"]}
    if kind == "scenarios":
        P.oed_eig_designs(st["ctx"], st["H_rec"], 0, st["mask"], st["w"], lo, hi, st["eig"], n_bad=st["n_bad"])
        out["H_rec"] = st["H_rec"]
        return out
    if kind == "study":
        P.oed_eig_subset(st["ctx"], st["H"], st["w"], lo, hi, PAPER_UNKNOWN, st["eig"], dkl=st["dkl"], n_bad=st["n_bad"])
    else:
        P.oed_eig(st["ctx"], st["H"], st["w"], lo, hi, st["eig"], dkl=st["dkl"], n_bad=st["n_bad"])
    out["dkl"] = st["dkl"]
    if kind == "windows":
        out["H_rec"] = st["H_rec"]
    return out


def work(case):
    """Bytes: inputs read once and outputs written once.  Flops: 33 per cell-update (the
    operator with shared differences), 98 per seismogram row of a Hessian, about 250 per 7x7
    log-determinant, three per squared difference of the double loop."""
    kind, n = case["kind"], case["n"]
    if kind == "designs":
        nd = 10 * case["per_k"]
        return {"bytes": 8.0 * n * case["nrec"] * 28 + nd * (case["nrec"] + 12.0) + 8.0 * n,
                "flops": n * nd * (28 * 5.5 + 250.0)}
    D = (case["nsteps"] + 1) * case["nrec"] * 2
    if kind == "dlmc":
        return {"bytes": 8.0 * (2 * n + case["m"]) * D + 8.0 * n, "flops": 3.0 * n * case["m"] * D}
    step = 33.0 * case["nx"] * case["nz"] * case["nsteps"]
    if kind == "forward":
        return {"bytes": n * (56.0 + 8 * D), "flops": n * step}
    per = 15 if case["jac"] == "pairs" else 7
    node = per * step + 98.0 * D + 250
    out = 8.0 * (7 + 49 + 2)
    if kind == "map":
        node = (case["iters"] + 1) * ((per + 2) * step + 98.0 * D)
        out += 8.0 * (14 + D)
    if kind in ("windows", "scenarios"):
        out += 8.0 * 28 * case["nrec"] * len(_win_levels(case))
    if kind == "scenarios":
        node += 36 * (28 * 12 + 250.0)
    return {"bytes": n * out, "flops": n * node}


# ------------------------------------------------- the same in 64 bits, plain torch / numpy

def _weight_polynomials():
    """The regularised delta and delta' at the six nodes k-2..k+3 as polynomials in the offset
    a = (x_s - x_k) / h, coefficients in ascending powers (times 1/h and 1/h^2)."""
    Pq = np.array([0, 0, 0, 0, 0, 5 / 3, -7 / 24, -17 / 12, 9 / 8, -1 / 4])
    R = np.array([0, 0, 0, 0, -25 / 12, -3 / 4, 59 / 12, -4, 1, 0])
    d = np.zeros((6, 10))
    d[:, :5] = [[0, 1 / 12, -1 / 24, -1 / 12, -19 / 24], [0, -2 / 3, 2 / 3, 1 / 6, 4], [1, 0, -5 / 4, 0, -97 / 12],
                [0, 2 / 3, 2 / 3, -1 / 6, 49 / 6], [0, -1 / 12, -1 / 24, 1 / 12, -33 / 8], [0, 0, 0, 0, 5 / 6]]
    p = np.zeros((6, 10))
    p[:, :4] = [[-1 / 12, 1 / 12, 1 / 4, 2 / 3], [2 / 3, -4 / 3, -1 / 2, -7 / 2], [0, 5 / 2, 0, 22 / 3],
                [-2 / 3, -4 / 3, 1 / 2, -23 / 3], [1 / 12, 1 / 12, -1 / 4, 4], [0, 0, 0, -5 / 6]]
    k = np.array([1, -5, 10, -10, 5, -1])[:, None]
    return d + k * Pq, p + k * R


def _weights(x, h, order):
    """order-th x_s-derivative of the delta and delta' weights of positions x[n]: [n][6] each,
    and the node index of the first weight."""
    q = x / h
    k = np.floor(q)
    a = (q - k)[:, None]
    out = []
    for pol, e in zip(_weight_polynomials(), (1, 2)):
        rows = [np.polynomial.polynomial.polyder(r, order) if order else r for r in pol]
        out.append(np.concatenate([np.polynomial.polynomial.polyval(a, r) for r in rows], axis=1) / h ** (e + order))
    return out[0], out[1], k.astype(np.int64) - 2


def _patch(case, th, ox=0, oz=0, moment=None):
    """Force densities [n][2][6][6] (component, depth, x) and corners of M grad(delta), with the
    ox-th / oz-th derivatives in x_s / z_s; moment: only that moment's unit term."""
    dx, px, i0 = _weights(th[:, 0], case["h"], ox)
    dz, pz, j0 = _weights(th[:, 1], case["h"], oz)
    m = [th[:, j] if moment is None else np.full(th.shape[0], float(moment == j)) for j in (4, 5, 6)]
    a, b = dz[:, :, None] * px[:, None, :], pz[:, :, None] * dx[:, None, :]
    m = [v[:, None, None] for v in m]
    return np.stack([m[0] * a + m[1] * b, m[1] * a + m[2] * b], axis=1), i0, j0


def _time(case, th, part="S"):
    """S(t_m) [n][nsteps] or one of its derivatives in t_s (t) and omega_s (w)."""
    u = np.arange(case["nsteps"])[None, :] * case["dt"] - th[:, 2:3]
    w = th[:, 3:4]
    S = w / math.sqrt(2 * math.pi) * np.exp(-0.5 * (w * u) ** 2)
    Lt, Lw = w * w * u, 1 / w - w * u * u
    return S * {"S": 1.0, "t": Lt, "w": Lw, "tt": Lt * Lt - w * w, "tw": Lt * Lw + 2 * w * u,
                "ww": Lw * Lw - 1 / (w * w) - u * u}[part]


def _solve(case, terms):
    """Seismograms [nsolve][nlev][nrec][2] of solves whose forcing is the sum of the terms, each
    (patch [nsolve][2][6][6], i0, j0, S [nsolve][nsteps]), by the leap-frog scheme."""
    nx, nz, h, dt = case["nx"], case["nz"], case["h"], case["dt"]
    lay = np.array(MEDIA[case["medium"]])
    l = np.searchsorted(lay[:, 0], np.arange(nz) * h, side="right") - 1
    vp, vs, rho = lay[l, 1], lay[l, 2], lay[l, 3]
    mu, lam = rho * vs ** 2, rho * (vp ** 2 - 2 * vs ** 2)
    pw, r = lam + 2 * mu, dt * dt / rho

    def rows(v):
        return torch.tensor(v[:-1, None], dtype=torch.float64, device=DEV)

    def dn(v):   # value on the row above
        return np.concatenate([v[:1], v[:-1]])

    def up(v):   # value on the row below
        return np.concatenate([v[1:], v[-1:]])

    q = r / (h * h)
    top = np.arange(nz) == 0
    half = np.where(top, 2.0, 1.0)      # the surface row's quadrature weight is one half
    own = np.where(top, 1.0, -1.0)      # and its cross terms take the row itself for the row above
    K = []
    for a, b, c in ((pw, mu, lam), (mu, pw, None)):
        # (second difference, south, north, cross south, cross north) of u_x, then of u_z
        s1, s0 = (lam, mu) if c is not None else (mu, lam)
        K.append([rows(v) for v in (
            q * a, half * q * 0.5 * (b + up(b)), np.where(top, 0.0, -q * 0.5 * (dn(b) + b)),
            half * q / 4 * (s1 + up(s0)), half * q / 4 * (own * np.where(top, s0, dn(s0)) - s1))])
    cp = [torch.tensor(v * dt / h, device=DEV) for v in (vp, vs)]
    ns = terms[0][0].shape[0]
    rec = torch.tensor(_receivers(case), device=DEV)
    g = torch.zeros((ns, case["nsteps"] + 1, rec.numel(), 2), dtype=torch.float64, device=DEV)
    f = [torch.zeros((ns, nz, nx), dtype=torch.float64, device=DEV) for _ in range(4)]
    cur, old = f[:2], f[2:]
    force = []
    for W, i0, j0, S in terms:
        jj = j0[:, None, None] + np.arange(6)[None, :, None]
        ii = i0[:, None, None] + np.arange(6)[None, None, :]
        at = torch.tensor((np.arange(ns)[:, None, None] * nz + jj) * nx + ii, device=DEV).flatten()
        W = W * r[jj[:, None] + 0 * ii[:, None]]
        force.append((at, [torch.tensor(W[:, k], device=DEV).flatten(1) for k in (0, 1)],
                      torch.tensor(S, device=DEV)))
    for m in range(case["nsteps"]):
        for k in (0, 1):
            g[:, m, :, k] = cur[k][:, 0, rec]
        cross = [u[:, :, 2:] - u[:, :, :-2] for u in cur]
        for k in (0, 1):
            u, c = cur[k], cur[k][:, :-1, 1:-1]
            axx, vs_, vn, ds, dn_ = K[k]
            new = old[k][:, :-1, 1:-1]
            torch.sub(c, new, out=new)
            d1 = u[:, :-1, 1:] - u[:, :-1, :-1]
            new.addcmul_(axx, d1[:, :, 1:] - d1[:, :, :-1])
            dv = u[:, 1:, 1:-1] - c
            x = cross[1 - k]
            new.addcmul_(vs_, dv).addcmul_(ds, x[:, 1:])
            new[:, 1:].addcmul_(vn[1:], dv[:, :-1]).addcmul_(dn_[1:], x[:, :-2])
            new[:, :1].addcmul_(dn_[:1], x[:, :1])
            new.add_(c)
            o, ca, cb = old[k], cp[k], cp[1 - k]
            o[:, -1, 1:-1] = u[:, -1, 1:-1] + cb[-1] * (u[:, -2, 1:-1] - u[:, -1, 1:-1])
            o[:, :, 0] = u[:, :, 0] + ca * (u[:, :, 1] - u[:, :, 0])
            o[:, :, -1] = u[:, :, -1] + ca * (u[:, :, -2] - u[:, :, -1])
            for at, W, S in force:
                o.view(-1).index_add_(0, at, (W[k] * S[:, m:m + 1]).flatten())
        cur, old = old, cur
    for k in (0, 1):
        g[:, -1, :, k] = cur[k][:, 0, rec]
    return g


def _seismograms(case, th):
    """Seismograms of parameter vectors th[n][7], in groups that keep the fields small."""
    step = max(1, int(2e8 / (case["nx"] * case["nz"])))
    out = []
    for a in range(0, th.shape[0], step):
        t = th[a:a + step]
        out.append(_solve(case, [(*_patch(case, t), _time(case, t))]))
    return torch.cat(out)


def _jacobian(case, th):
    """Jacobian columns [n][7][nlev][nrec][2]: central differences with the step of the Hessian
    call, as solves driven by the difference of the two forcings; or sensitivity solves."""
    lo, hi = (np.array(v) for v in PRIORS[case["prior"]])
    d = REL_STEP * (hi - lo)
    cols = []
    for j in range(7):
        if case["jac"] == "sensitivity":
            W = _patch(case, th, ox=int(j == 0), oz=int(j == 1), moment=j if j >= 4 else None)
            terms = [(*W, _time(case, th, {2: "t", 3: "w"}.get(j, "S")))]
        else:
            terms = []
            for sign in (1.0, -1.0):
                t = th.copy()
                t[:, j] += sign * d[j]
                W, i0, j0 = _patch(case, t)
                terms.append((W * (sign / (2 * d[j])), i0, j0, _time(case, t)))
        cols.append(_solve(case, terms))
    return torch.stack(cols, dim=1)


def _gain(H, logvol):
    """D_KL-hat of a batch of Hessians [..., k, k] from the scaled Cholesky factor."""
    k = H.shape[-1]
    d = torch.diagonal(H, dim1=-2, dim2=-1)
    s = d.sqrt()
    Ht = H / (s[..., :, None] * s[..., None, :])
    L = {}
    ld = d.log().sum(-1)
    for j in range(k):
        v = Ht[..., j, j] - sum((L[j, c] ** 2 for c in range(j)), torch.zeros_like(Ht[..., 0, 0]))
        L[j, j] = v.sqrt()
        ld = ld + v.log()
        for i in range(j + 1, k):
            L[i, j] = (Ht[..., i, j] - sum((L[i, c] * L[j, c] for c in range(j)), torch.zeros_like(v))) / L[j, j]
    return 0.5 * ld - 0.5 * k * (math.log(2 * math.pi) + 1) + logvol


def _full(h28):
    """Symmetric 7x7 matrices from the packed upper triangle."""
    iu = torch.triu_indices(7, 7, device=DEV)
    H = torch.empty((*h28.shape[:-1], 7, 7), dtype=torch.float64, device=DEV)
    H[..., iu[0], iu[1]] = h28
    H[..., iu[1], iu[0]] = h28
    return H


def _design_gains(H_rec, mask, logvol):
    """EIG of every design: mean over nodes of the gain of the masked sum of partial Hessians."""
    n, nd = H_rec.shape[0], mask.shape[0]
    out = torch.empty(nd, dtype=torch.float64, device=DEV)
    step = max(1, int(2e6 / n))
    m = torch.tensor(mask, dtype=torch.float64, device=DEV)
    for a in range(0, nd, step):
        h = torch.einsum("dr,nrk->dnk", m[a:a + step], H_rec)
        out[a:a + step] = _gain(_full(h), logvol).mean(1)
    return out


def _newton(case, th, y):
    """Newton iterations on the cost over the unknowns with H_1 + H_II, the second-derivative
    terms from solves driven by the forcing's second derivatives (the scheme is linear)."""
    lo, hi = (np.array(v) for v in PRIORS[case["prior"]])
    F = list(PAPER_UNKNOWN)
    n = th.shape[0]
    for it in range(case["iters"] + 1):
        w = (y - _seismograms(case, th)) / case["sigma"] ** 2
        J = _jacobian(case, th)
        H = torch.einsum("ajmrc,akmrc->ajk", J, J) / case["sigma"] ** 2
        grad = -torch.einsum("ajmrc,amrc->aj", J, w)
        for p in range(7):
            for q in range(p, 7):
                if p >= 4:
                    continue
                part = "".join(sorted(("t" if j == 2 else "w") for j in (p, q) if j in (2, 3))) or "S"
                W = _patch(case, th, ox=(p == 0) + (q == 0), oz=(p == 1) + (q == 1), moment=q if q >= 4 else None)
                v = torch.einsum("amrc,amrc->a", _solve(case, [(*W, _time(case, th, part))]), w)
                H[:, p, q] -= v
                if q != p:
                    H[:, q, p] -= v
        if it == case["iters"]:
            return th, H, grad
        Hf = H[:, F][:, :, F]
        s = torch.diagonal(Hf, dim1=-2, dim2=-1).clamp_min(0).sqrt()
        Ht = Hf / (s[:, :, None] * s[:, None, :])
        ok = torch.linalg.cholesky_ex(torch.nan_to_num(Ht, nan=-1.0)).info == 0
        ok &= (torch.diagonal(Hf, dim1=-2, dim2=-1) > 0).all(-1)
        eye = torch.eye(len(F), dtype=torch.float64, device=DEV)
        step = torch.linalg.solve(torch.where(ok[:, None, None], Ht, eye), -grad[:, F] / s) / s
        step = torch.where(ok[:, None], step, torch.zeros_like(step)).cpu().numpy()
        th = th.copy()
        moved = np.minimum(np.maximum(th[:, F] + step, lo[F]), hi[F])
        th[:, F] = np.where(ok.cpu().numpy()[:, None], moved, th[:, F])
    raise AssertionError("unreachable")


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    lo, hi = (np.array(v) for v in PRIORS[case.get("prior", "half_plane")])
    logvol = float(np.sum(np.log(hi - lo)))
    if kind == "designs":
        H_rec = _partial_hessians(case, seed)[:, :, case["win"]]
        return {"eig": _design_gains(H_rec, _subset_designs(case, seed), logvol), "n_bad": None}
    if kind == "dlmc":
        m = case["m"]
        g = _seismograms(case, np.concatenate([_thetas(case, n, seed), _thetas(case, m, seed + 7919)])).flatten(1)
        eps = _noise(case, (n, g.shape[1]), seed)
        y, s2 = g[:n] + eps, 2 * case["sigma"] ** 2
        step = max(1, int(1e8 / (m * g.shape[1])))
        d2 = torch.cat([((y[a:a + step, None] - g[None, n:]) ** 2).sum(-1) for a in range(0, n, step)])
        ev = torch.logsumexp(-d2 / s2, dim=1) - math.log(m)
        return {"log_ev": ev, "eig": (-(eps ** 2).sum(-1) / s2 - ev).mean().reshape(1)}
    th = _thetas(case, n, seed)
    if kind == "forward":
        if case["nx"] * case["nz"] * case["nsteps"] * n > 9e10:
            return None
        return {"g": _seismograms(case, th)}
    if kind == "map":
        y = _seismograms(case, th)
        th, H, grad = _newton(case, th, y + _noise(case, tuple(y.shape), seed))
        return {"theta": torch.tensor(th, device=DEV), "H": H, "grad": grad, "status": None}
    if 7 * case["nx"] * case["nz"] * case["nsteps"] * n > 9e10:
        return None   # about 20 seconds of plain 64-bit time steps
    hw, tot = [], []
    ends = [0] + (_win_levels(case) if kind in ("windows", "scenarios") else [])
    iu = torch.triu_indices(7, 7, device=DEV)
    step = max(1, int(1e8 / (7 * max(case["nx"] * case["nz"], (case["nsteps"] + 1) * case["nrec"] * 2))))
    for a in range(0, n, step):
        J = _jacobian(case, th[a:a + step]) / case["sigma"]
        tot.append(torch.einsum("ajmrc,akmrc->ajk", J, J))
        if len(ends) > 1:
            w = [torch.einsum("ajmrc,akmrc->arjk", J[:, :, :e], J[:, :, :e]) for e in ends[1:]]
            hw.append(torch.stack(w, dim=2)[..., iu[0], iu[1]])
        del J
    H = torch.cat(tot)
    if kind == "study":
        F = list(PAPER_UNKNOWN)
        dkl = _gain(H[:, F][:, :, F], float(np.sum(np.log((hi - lo)[F]))))
    else:
        dkl = _gain(H, logvol)
    if kind == "host":
        return {"eig": float(dkl.mean()), "dkl": dkl, "n_bad": None}
    out = {"H": H, "status": None, "eig": dkl.mean().reshape(1), "n_bad": None}
    if kind == "scenarios":
        out["H_rec"] = torch.cat(hw)
        out["eig"] = _design_gains(out["H_rec"][:, :, 0], _line_designs(), logvol)
        return out
    out["dkl"] = dkl
    if kind == "windows":
        out["H_rec"] = torch.cat(hw)
    return out
