"""The FP64 kernels on batches that give their threads several rows.

k_step64 and k_adjoint64 cut a column into segments of one row where a batch fits the FP64
pipes in one round, and of up to eight and four rows where it does not.  The node updates are
the same operations in the same order at every segment length, so each solve of a large batch
equals the solve on its own (one-row segments) bit for bit: at row counts that the segments
do not divide, even and odd widths, the smallest grid, homogeneous and layered.  One solve of
a batch against the FP64 oracle besides: 1e-12 of the peak for seismograms (60 steps of a
stable scheme at 2^-53 each), 1e-9 of the Gauss-Newton scale (times the norm of the residual)
for the dual solve.
"""
import math

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LAYERS = ((0.0, 1800.0, 1000.0, 2100.0), (40.0, 2600.0, 1500.0, 2300.0), (120.0, 4000.0, 2300.0, 2700.0))


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1502_07873_gb300 as P
    return P


def _segment(columns, nz, zs, per, once):
    """Longest and shortest segment of the rule in stencil.cu on a chip of 152 SMs."""
    best = None
    for r in range(zs, 0, -1):
        nseg = -(-nz // r)
        rows, warps = -(-nz // nseg), columns * nseg / (32 * 608)
        cost = max(1.0, 0.5 * (warps + math.ceil(warps))) * (per * rows + once) + 8 * rows
        if best is None or cost < best[0]:
            best = (cost, nseg)
    return -(-nz // best[1]), nz // best[1]


def _workload(nx, nz, layers):
    return W.tiny(nx=nx, nz=nz, h=20.0, nsteps=60, nrec=min(5, nx), layers=layers)


def _thetas(w, n, seed):
    rng = np.random.default_rng(seed)
    x = 3.0 + rng.random(n) * max(0.0, w.nx - 8.1)
    z = 2.0 + rng.random(n) * max(0.0, w.nz - 7.1)
    m = 1e13 + 9e13 * rng.random((n, 3))
    return np.column_stack([x * w.h, z * w.h, 0.02 * rng.random(n), 4.0 + 4.0 * rng.random(n), m])


def _forward(P, ctx, w, th):
    g = torch.empty((th.shape[0], w.nlevels, w.nrec, 2), dtype=torch.float64, device=DEV)
    P.oed_forward(ctx, torch.tensor(th, device=DEV), g)
    torch.cuda.synchronize()
    return g


def _picks(n):
    return sorted({0, 1, n // 3, n // 2, n - 2, n - 1} | set(np.random.default_rng(n).integers(0, n, 6).tolist()))


@pytest.mark.parametrize("nx,nz,n,rows", [
    (8, 8, 3000, {2: (2, 2), 4: (2, 2), 8: (2, 2)}), (9, 9, 3000, {2: (2, 1), 4: (3, 3), 8: (3, 3)}),
    (33, 17, 60, {2: (1, 1), 4: (1, 1), 8: (1, 1)}), (33, 17, 1500, {2: (2, 1), 4: (3, 2), 8: (6, 5)}),
    (41, 29, 500, {2: (2, 1), 4: (3, 2), 8: (6, 5)}), (64, 41, 500, {2: (2, 1), 4: (3, 2), 8: (7, 6)}),
    (81, 41, 60, {2: (2, 1), 4: (3, 2), 8: (3, 2)}), (101, 76, 240, {2: (2, 2), 4: (4, 4), 8: (7, 6)}),
])
@pytest.mark.parametrize("layers", [W.HOMOGENEOUS, LAYERS], ids=["homogeneous", "layered"])
def test_step64_rows_per_thread(P, oracle, nx, nz, n, rows, layers):
    for zs, r in rows.items():   # the batch does what the name says
        assert _segment((nx + 1) // 2 * n, nz, zs, 23, 10) == r
    assert _segment((nx + 1) // 2, nz, 8, 23, 10) == (1, 1)
    w = _workload(nx, nz, layers)
    th = _thetas(w, n, nx)
    one = P.Context(P.problem_from_workload(w, P.OED_FP64), max_solves=1)
    one.set_tuning(0, 4, 4)
    picks = _picks(n)
    ref = torch.cat([_forward(P, one, w, th[k:k + 1]) for k in picks])
    one.close()
    assert float(ref.abs().max()) > 0
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP64), max_solves=n)
    for zs in rows:
        for wz in (1, 8):
            ctx.set_tuning(0, zs, wz)
            assert torch.equal(_forward(P, ctx, w, th)[picks], ref), (zs, wz)
    ctx.close()
    o = oracle.forward(oracle.Grid.from_workload(w), th[picks[2]])
    assert np.max(np.abs(ref[2].cpu().numpy() - o)) <= 1e-12 * np.max(np.abs(o))


@pytest.mark.parametrize("nx,nz,n,rows", [
    (8, 8, 1000, (2, 2)), (9, 9, 3000, (3, 3)), (33, 17, 100, (1, 1)), (33, 17, 240, (2, 1)), (41, 29, 500, (3, 2)),
    (64, 41, 240, (4, 3)), (81, 41, 100, (3, 2)), (101, 76, 60, (4, 4)),
])
@pytest.mark.parametrize("layers", [W.HOMOGENEOUS, LAYERS], ids=["homogeneous", "layered"])
def test_adjoint64_rows_per_thread(P, oracle, nx, nz, n, rows, layers):
    assert _segment(nx * n, nz, 4, 16, 8) == rows
    assert _segment(nx, nz, 4, 16, 8) == (1, 1)
    w = _workload(nx, nz, layers)
    th = _thetas(w, n, nz)
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP64), max_solves=n)
    ctx.set_tuning(0, 4, 4)
    y = _forward(P, ctx, w, th)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n)
    sigma = float(y.abs().max()) * 0.1
    y += sigma * torch.randn(y.shape, dtype=torch.float64, device=DEV, generator=gen)

    def dual(c, t, data):
        H = torch.zeros((t.shape[0], 7, 7), dtype=torch.float64, device=DEV)
        gr = torch.empty((t.shape[0], 7), dtype=torch.float64, device=DEV)
        P.oed_hessian_ii(c, torch.tensor(t, device=DEV), data, sigma, H, grad=gr)
        torch.cuda.synchronize()
        return H, gr

    H, gr = dual(ctx, th, y)
    ctx.close()
    assert bool(torch.isfinite(H).all()) and float(H.abs().max()) > 0
    one = P.Context(P.problem_from_workload(w, P.OED_FP64), max_solves=1)
    one.set_tuning(0, 4, 4)
    picks = _picks(n)
    for k in picks:
        H1, g1 = dual(one, th[k:k + 1], y[k:k + 1].contiguous())
        assert torch.equal(H[k], H1[0]) and torch.equal(gr[k], g1[0]), k
    one.close()
    if nx < 33:
        return
    k = picks[2]
    G = oracle.Grid.from_workload(w)
    data = y[k].cpu().numpy()
    H2, g2 = oracle.hessian_ii(G, th[k], data, sigma)
    d = np.sqrt(np.diag(oracle.node_hessian_sensitivity(G, th[k], sigma)))
    rnorm = np.sqrt(np.sum((data - oracle.forward(G, th[k])) ** 2)) / sigma
    assert np.max(np.abs(H[k].cpu().numpy() - H2) / np.outer(d, d)) <= 1e-9 * max(1.0, rnorm)
    assert np.max(np.abs(gr[k].cpu().numpy() - g2) / (d * rnorm)) <= 1e-9
