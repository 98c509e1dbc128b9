"""The multi-step strip kernel (four leap-frog steps per pass, Eq. Full_Disc) at the edges of
its strips, bands, chunks and coefficient runs: its seismograms equal the register
streaming kernel's bit for bit.  Grids wider than 1216 columns do not fit on chip at any
depth, so few rows suffice.  Widths around a multiple of the 56-column strip (even and
odd, so with and without a ghost column), every remainder of the step count by four,
receivers on strip edges, repeated and more than a warp of them, sources whose patches
touch the surface, the sides and the bottom, one solve and several (one band and more),
and media with an interface at almost every row.
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
    for k in range(n):
        vs = 1000.0 + 900.0 * rng.random()
        out.append((z, 1.8 * vs, vs, 2200.0 + 500.0 * rng.random()))
        z += h * int(rng.integers(1, 5))
    return tuple(out)


@pytest.mark.parametrize("nx,nz,nsteps,nlayer,nsolve", [
    (1232, 33, 4, 1, 1), (1233, 34, 5, 1, 3), (1231, 35, 6, 3, 2), (1288, 40, 7, 12, 5),
    (1234, 41, 1, 1, 2), (1287, 97, 23, 1, 2), (1289, 160, 40, 30, 1), (1230, 64, 30, 1, 60),
])
def test_strip_kernel_bitwise(P, nx, nz, nsteps, nlayer, nsolve):
    h = 5.0
    layers = W.HOMOGENEOUS if nlayer == 1 else _layers(nlayer, h)
    w = W.tiny(nx=nx, nz=nz, h=h, nsteps=nsteps, layers=layers)
    rec = [0, 1, 55, 56, 57, 111, 112, 560, nx // 2, nx - 2, nx - 1, 56, 0] + list(range(3, nx, 41))
    # corners of the source patch: left, right, surface, bottom and strip edges, then spread
    rng = np.random.default_rng(nx + nz)
    at = [(3.3, 2.4), (nx - 5.5, nz - 5.2), (57.9, 2.0), (112.0, nz - 5.5), (nx / 2, nz / 2)]
    at += [(3.0 + rng.random() * (nx - 9), 2.0 + rng.random() * (nz - 8)) for _ in range(nsolve)]
    th = np.array([[x * h, z * h, 0.0, 6.0, 6e13, 3e13, 9e13] for x, z in at[:nsolve]])
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32, rec_ix=rec), max_solves=nsolve)
    g = {}
    for tune in ((0, 4, 4), (-2, 4, 4)):
        ctx.set_tuning(*tune)
        g[tune[0]] = torch.full((nsolve, nsteps + 1, len(rec), 2), float("nan"), dtype=torch.float64, device=DEV)
        P.oed_forward(ctx, torch.tensor(th, device=DEV), g[tune[0]])
    torch.cuda.synchronize()
    ctx.close()
    assert bool(torch.isfinite(g[0]).all())
    assert nsteps < 4 or float(g[0].abs().max()) > 0
    assert torch.equal(g[0], g[-2])
