"""Launch shapes that depend on sizes.

The resident kernel plans several CTAs per SM when a launch has enough solves: with 1 and
with many solves its seismograms equal the register streaming kernel's bit for bit, on
grids that take one to six CTAs per SM, with layer interfaces inside and between the row
segments.  The FP64 step packs its threads densely over solves, row segments and column
pairs: every shape equals every other bit for bit and the FP64 oracle to rounding (1e-12
of the peak: a few hundred steps of a stable scheme at 2^-53 each), on the smallest grid, at
even and odd widths, with row counts that the segments do not divide.
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


def _thetas(nx, nz, h, n, seed):
    rng = np.random.default_rng(seed)
    x = 3.0 + rng.random(n) * max(0.0, nx - 8.1)
    z = 2.0 + rng.random(n) * max(0.0, nz - 7.1)
    m = 1e13 + 9e13 * rng.random((n, 3))
    return np.column_stack([x * h, z * h, 0.02 * rng.random(n), 4.0 + 4.0 * rng.random(n), m])


def _forward(P, ctx, th, w):
    g = torch.full((th.shape[0], w.nlevels, w.nrec, 2), float("nan"), dtype=torch.float64, device=DEV)
    P.oed_forward(ctx, torch.tensor(th, device=DEV), g)
    torch.cuda.synchronize()
    return g


LAYERS = ((0.0, 1800.0, 1000.0, 2100.0), (140.0, 2600.0, 1500.0, 2300.0), (150.0, 3000.0, 1700.0, 2500.0),
          (420.0, 4000.0, 2300.0, 2700.0))


@pytest.mark.parametrize("nx,nz,nsolve,clusters", [
    (61, 31, 1, (1, 2)), (61, 31, 1000, (1, 2)), (81, 41, 700, (1, 3)), (82, 42, 460, (1,)),
    (101, 76, 400, (1, 2)), (120, 61, 200, (1, 2)), (201, 101, 120, (2, 3)), (9, 8, 900, (1,)),
])
@pytest.mark.parametrize("layers", [W.HOMOGENEOUS, LAYERS], ids=["homogeneous", "layered"])
def test_resident_shapes_bitwise(P, nx, nz, nsolve, clusters, layers):
    h = 20.0
    w = W.tiny(nx=nx, nz=nz, h=h, nsteps=21, nrec=min(7, nx), layers=layers)
    th = _thetas(nx, nz, h, nsolve, seed=nx + nsolve)
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32), max_solves=nsolve)
    ctx.set_tuning(0, 4, 4)
    ref = _forward(P, ctx, th, w)
    assert float(ref.nan_to_num().abs().max()) > 0
    for C in clusters:
        ctx.set_tuning(C, 4, 4)
        assert torch.equal(_forward(P, ctx, th, w).nan_to_num(nan=-1.0), ref.nan_to_num(nan=-1.0)), C
    ctx.close()


@pytest.mark.parametrize("nx,nz,nsolve", [(8, 8, 3), (9, 9, 70), (33, 17, 1), (64, 41, 5), (81, 38, 9)])
@pytest.mark.parametrize("layers", [W.HOMOGENEOUS, LAYERS], ids=["homogeneous", "layered"])
def test_fp64_step_shapes(P, oracle, nx, nz, nsolve, layers):
    h = 20.0
    w = W.tiny(nx=nx, nz=nz, h=h, nsteps=60, nrec=min(7, nx), layers=layers)
    rec = [0, nx - 1, nx // 2, 0, 1]
    th = _thetas(nx, nz, h, nsolve, seed=nx)
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP64, rec_ix=rec), max_solves=nsolve)
    w.rec_ix = rec
    out = []
    for zs in (2, 4, 8):
        for wz in (1, 8):
            ctx.set_tuning(0, zs, wz)
            out.append(_forward(P, ctx, th, w).nan_to_num(nan=-1.0))
    ctx.close()
    assert all(torch.equal(o, out[0]) for o in out[1:])
    G = oracle.Grid(nx, nz, h, w.dt, w.nsteps, w.layers, rec)
    for k in range(min(nsolve, 4)):
        got, ref = out[0][k].cpu().numpy(), oracle.forward(G, th[k])
        if np.all(np.isfinite(ref)):
            assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), k
