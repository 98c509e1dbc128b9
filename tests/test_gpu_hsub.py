"""The Gauss-Newton sums' time sub-segments and their widening of FP32 samples.

How the levels are cut depends on the record's length, the receivers and the windows: however it
is cut, the receivers' last windows add up to H, and a window's partial sum equals the one taken
without the other windows.  Two orders of the same N = 2 nlev nrec products differ by at most
2 N 2^-53 sqrt(H_xx H_yy) (Cauchy-Schwarz on the absolute values), in FP64.

Scaling every moment by a power of two scales FP32 seismograms exactly, until they become
subnormal: then each step rounds to 2^-149, some 2^-141 after sixty steps, and a parameter whose
samples' root mean square is 2^-136 or more keeps H_xx to 2^-3 (taking a subnormal for a normal
number would raise it by 2^18).
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


def _problem(P, nrec, nsteps, prec):
    w = W.tiny(nx=41, nz=21, h=50.0, nsteps=nsteps, nrec=nrec)
    rng = np.random.default_rng(nrec + nsteps)
    lo, hi = np.array(w.prior_lo), np.array(w.prior_hi)
    return w, lo + (hi - lo) * (0.3 + 0.4 * rng.random((3, 7)))


def _hessian(P, ctx, w, th, lo, hi, wl=None):
    n = th.shape[0]
    H = torch.full((n, 7, 7), float("nan"), dtype=torch.float64, device=DEV)
    Hr = torch.full((n, w.nrec, len(wl or [1]), 28), float("nan"), dtype=torch.float64, device=DEV)
    P.oed_hessian(ctx, torch.tensor(th, device=DEV), lo, hi, w.rel_step, 0.1, H,
                  **(dict(win_levels=wl, H_rec=Hr) if wl else {}))
    torch.cuda.synchronize()
    return H.cpu().numpy(), Hr.cpu().numpy()


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("mode", ["PAIRS", "DIFFERENCE"])
@pytest.mark.parametrize("nrec,nsteps", [(1, 1), (1, 40), (2, 600), (7, 150), (33, 63), (41, 130)])
def test_segments_add_up(P, nrec, nsteps, mode, prec):
    w, th = _problem(P, nrec, nsteps, prec)
    ctx = P.Context(P.problem_from_workload(w, getattr(P, "OED_" + prec)), max_solves=45)
    ctx.jacobian = getattr(P, "OED_JAC_" + mode)
    L = w.nlevels
    H, _ = _hessian(P, ctx, w, th, w.prior_lo, w.prior_hi)
    iu = np.triu_indices(7)
    d = np.sqrt(np.einsum("nxx->nx", H))
    tol = 2 * 2 * L * nrec * 2.0 ** -53 * (d[:, :, None] * d[:, None, :])[:, iu[0], iu[1]]
    last = {}
    for wl in ([L], sorted({max(1, L // 3), L}), sorted({max(1, L * k // 15) for k in range(1, 16)})):
        H2, Hr = _hessian(P, ctx, w, th, w.prior_lo, w.prior_hi, wl)
        assert np.all(np.isfinite(Hr))
        assert np.all(np.abs(H2 - H)[:, iu[0], iu[1]] <= tol)
        assert np.all(np.abs(Hr[:, :, -1].sum(1) - H[:, iu[0], iu[1]]) <= tol)
        for k, m in enumerate(wl):
            if m in last:
                assert np.all(np.abs(Hr[:, :, k] - last[m]) <= tol[:, None])
            last[m] = Hr[:, :, k]
    ctx.close()


def test_subnormal_samples(P):
    w, th = _problem(P, 7, 60, "FP32")
    ctx = P.Context(P.problem_from_workload(w, P.OED_FP32), max_solves=21)
    ctx.jacobian = P.OED_JAC_DIFFERENCE
    lo, hi = np.array(w.prior_lo), np.array(w.prior_hi)
    H, _ = _hessian(P, ctx, w, th, lo, hi)
    diag = np.einsum("nxx->nx", H)
    # H_xx = sum (g_x / 2 d_x)^2 / sigma^2
    rms = 2 * w.rel_step * (hi - lo) * 0.1 * np.sqrt(diag / (2 * w.nlevels * w.nrec))
    for e in (-100, int(np.floor(-130 - np.log2(rms.max())))):
        s = 2.0 ** e
        sc = np.array([1, 1, 1, 1, s, s, s])
        H2, _ = _hessian(P, ctx, w, th * sc, lo * sc, hi * sc)
        got = np.einsum("nxx->nx", H2) / np.array([s * s] * 4 + [1.0] * 3)
        if e == -100 and rms.min() * s > 2.0 ** -116:
            assert np.allclose(got, diag, rtol=1e-6)
        else:
            keep = rms * s >= 2.0 ** -136
            assert keep.any()
            assert np.all(np.abs(got - diag)[keep] <= diag[keep] / 8)
    ctx.close()
