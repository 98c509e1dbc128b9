"""The two-step TMA kernel (two leap-frog steps per pass, Eq. Full_Disc) at the edges of its
60-column tiles and 20-row bands: its seismograms equal the register streaming kernel's bit for bit,
on even and odd widths (a ghost column), one tile and several, fewer rows than a band, even and odd step
counts down to one (the last pass of an odd count takes one step), one solve and more than the
persistent CTAs take at once, media with an interface at almost every row, sources that
touch the surface, the sides and the bottom, repeated receivers, and on the replay of the
captured loop.  The autotuner times it beside the strip kernel, and whichever it takes gives the
same bits.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1502_07873_gb300 as P
    return P


def _layers(n, h):
    """n layers, one to four rows thick."""
    rng = np.random.default_rng(n)
    out, z = [], 0.0
    for _ in range(n):
        vs = 1000.0 + 900.0 * rng.random()
        out.append((z, 1.8 * vs, vs, 2200.0 + 500.0 * rng.random()))
        z += h * int(rng.integers(1, 5))
    return tuple(out)


def _thetas(w, n):
    rng = np.random.default_rng(n + w.nx)
    col = np.concatenate([[3.0, w.nx - 5.5, 60.0, 119.5, 62.25], 3.0 + rng.random(n) * (w.nx - 8.1)])[:n]
    row = np.concatenate([[2.0, w.nz - 5.25, 2.5, max(2.0, w.nz - 6.0), 3.0], 2.0 + rng.random(n) * (w.nz - 7.1)])[:n]
    m = 1e13 + 9e13 * rng.random((n, 3))
    return np.column_stack([col * w.h, row * w.h, 0.01 * rng.random(n), 5.0 + 4.0 * rng.random(n), m])


def _forward(P, ctx, th, w):
    g = torch.full((th.shape[0], w.nlevels, w.nrec, 2), float("nan"), dtype=torch.float64, device=DEV)
    P.oed_forward(ctx, torch.tensor(th, device=DEV), g)
    torch.cuda.synchronize()
    return g.nan_to_num(nan=-1.0)


@pytest.mark.parametrize("nx,nz,nsteps,nlayer,nsolve", [
    (1217, 9, 21, 1, 1), (1217, 8, 1, 2, 3), (1260, 20, 2, 1, 2), (1261, 21, 5, 9, 5), (1301, 41, 30, 12, 4),
    (1219, 40, 33, 20, 40), (801, 401, 12, 60, 2), (40, 4000, 9, 3, 5), (415, 801, 7, 1, 1),
])
def test_bitwise(P, nx, nz, nsteps, nlayer, nsolve):
    h = 20.0
    w = W.tiny(nx=nx, nz=nz, h=h, nsteps=nsteps, nrec=12, layers=_layers(nlayer, h))
    rec = sorted({0, 1, min(59, nx - 2), min(60, nx - 2), nx // 2, nx - 2, nx - 1}) + [0]
    w.rec_ix = rec
    th = _thetas(w, nsolve)
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32, rec_ix=rec), max_solves=nsolve)
    assert ctx.resident_min_cluster == 0   # the grid does not fit on chip
    ctx.set_tuning(0, 4, 4)
    ref = _forward(P, ctx, th, w)
    assert nsteps < 5 or float(ref.abs().max()) > 0
    ctx.set_tuning(-3, 4, 4)
    assert ctx.tuning[0] == -3
    for _ in range(2):   # the second call replays the captured time loop
        assert torch.equal(_forward(P, ctx, th, w), ref)
    assert ctx.autotune(nsolve)[0] in (0, -1, -2, -3)
    assert torch.equal(_forward(P, ctx, th, w), ref)
    ctx.close()


def test_hessians(P):
    w = W.tiny(nx=1261, nz=41, h=20.0, nsteps=60, nrec=8, layers=W.THREE_LAYER)
    th = _thetas(w, 4)
    lo, hi = th.min(0) * 0.9 - 1e-3, th.max(0) * 1.1 + 1e-3
    H = []
    for tune in ((0, 4, 4), (-3, 4, 4)):
        ctx = P.Context(P.problem_from_workload(w, P.OED_FP32), max_solves=21)   # chunks of three nodes and of one
        ctx.jacobian = P.OED_JAC_DIFFERENCE
        ctx.set_tuning(*tune)
        H.append(torch.zeros((4, 7, 7), dtype=torch.float64, device=DEV))
        P.oed_hessian(ctx, torch.tensor(th, device=DEV), lo, hi, 1e-4, 0.1, H[-1])
        torch.cuda.synchronize()
        ctx.close()
    assert torch.equal(H[0].nan_to_num(nan=-1.0), H[1].nan_to_num(nan=-1.0)) and float(H[0].nan_to_num().abs().max()) > 0


@pytest.mark.parametrize("nx,nz,prec", [(401, 201, 0), (1301, 20, 1)])
def test_refused(P, nx, nz, prec):
    w = W.tiny(nx=nx, nz=nz, h=20.0, nsteps=10, nrec=4)
    ctx = P.Context(P.problem_from_workload(w, prec), max_solves=2)
    with pytest.raises(P.OedError):
        ctx.set_tuning(-3, 4, 4)
    ctx.close()


def test_large_batches_take_the_strip_kernel(P):
    """Without a probe, so that other work on the device cannot change the choice."""
    w = W.tiny(nx=801, nz=401, h=2.5, nsteps=8, nrec=4, layers=W.THREE_LAYER)
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32), max_solves=14)
    assert ctx.autotune(14)[0] == -2
    ctx.close()
