"""The resident kernel's padded rows and segments and its edge warp: seismograms equal the
register streaming kernel's bit for bit on widths of every kind modulo four, with row segments of
two to 32 rows (an interface in the first, the last and the 32nd row), slabs of more than 64 rows,
more than 96 receivers, and the receivers on the side columns.
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


@pytest.mark.parametrize("nx,nz,nsolve,clusters", [
    (60, 31, 700, (1, 2, 3)), (62, 33, 500, (1, 4)), (65, 96, 40, (3, 4)), (66, 64, 30, (2, 8)),
    (33, 100, 200, (1, 2)), (8, 130, 9, (1, 2)), (102, 76, 300, (1, 2)), (203, 60, 30, (1, 2, 7)),
    (404, 40, 9, (2, 3)), (121, 61, 170, (1, 5)),
])
def test_padded_slots_bitwise(P, nx, nz, nsolve, clusters):
    h, nsteps = 20.0, 25
    # the elastic row 31 below a segment's first is the 32nd that it can hold
    layers = ((0.0, 1800.0, 1000.0, 2100.0), (1.2 * h, 2000.0, 1100.0, 2200.0), (31.2 * h, 2600.0, 1500.0, 2300.0),
              ((nz - 2.5) * h, 4000.0, 2300.0, 2700.0))
    w = W.tiny(nx=nx, nz=nz, h=h, nsteps=nsteps, nrec=min(7, nx), layers=layers if nz > 34 else layers[:2])
    rec = [0, nx - 1, 1, nx - 2] + [k % nx for k in range(100)]
    rng = np.random.default_rng(nx + nz)
    x = 3.0 + rng.random(nsolve) * max(0.0, nx - 8.1)
    z = 2.0 + rng.random(nsolve) * min(max(0.0, nz - 7.1), 9.0)
    th = np.column_stack([x * h, z * h, 0.02 * rng.random(nsolve), 4.0 + 4.0 * rng.random(nsolve),
                          1e13 + 9e13 * rng.random((nsolve, 3))])
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32, rec_ix=rec), max_solves=nsolve)
    out = {}
    for C in (0,) + clusters:
        ctx.set_tuning(C, 4, 4)
        g = torch.full((nsolve, nsteps + 1, len(rec), 2), float("nan"), dtype=torch.float64, device=DEV)
        P.oed_forward(ctx, torch.tensor(th, device=DEV), g)
        torch.cuda.synchronize()
        out[C] = g.nan_to_num(nan=-1.0)
        assert torch.equal(out[C], out[0]), C
    ctx.close()
    assert float(out[0].abs().max()) > 0
