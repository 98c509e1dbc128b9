"""The screened double loop: pairs of samples are left out of the FP64 sums only where they
cannot matter, so log_ev equals the plain FP64 formula to rounding (1e-12, a few hundred
FP64 operations per distance and at most a few thousand per sum) for every mix of near and
far samples, odd and long data rows, unaligned data, one sample, and a full list of kept
samples; non-finite data give what they gave: NaN where an inner sample is NaN, -inf for a
row of NaN, and nothing from a sample at infinite distance."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1502_07873_gb300 as P
    return P


def _plain(y, gi, sigma):
    d2 = torch.cat([((y[k:k + 1] - gi) ** 2).sum(-1)[None] for k in range(y.shape[0])])
    return torch.logsumexp(-d2 / (2 * sigma ** 2), dim=1) - math.log(gi.shape[0])


def _run(P, go, eps, gi, sigma):
    log_ev = torch.full((go.shape[0],), 7.0, dtype=torch.float64, device=DEV)
    eig = torch.zeros(1, dtype=torch.float64, device=DEV)
    P.oed_dlmc(go, eps, gi, sigma, log_ev, eig)
    torch.cuda.synchronize()
    return log_ev, eig


@pytest.mark.parametrize("N,M,D,spread,sigma", [
    (1, 1, 1, 1.0, 0.1), (3, 1, 7, 1.0, 0.5), (65, 129, 31, 0.02, 0.01), (64, 64, 32, 5.0, 0.01),
    (70, 3000, 33, 0.001, 0.01), (9, 5000, 64, 0.3, 0.01), (130, 257, 200, 0.03, 0.01), (5, 40, 12290, 0.01, 0.01),
    (33, 700, 20, 1e-30, 1e-31), (33, 700, 20, 1e30, 1e29), (40, 90, 16, 1e6, 1e-3),
])
def test_screened_equals_plain(P, N, M, D, spread, sigma):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N + M + D)
    rnd = lambda *s: torch.randn(s, dtype=torch.float64, device=DEV, generator=gen)
    base = spread * rnd(1, D) * 10
    # samples on a line through the data space, so rows have near and far neighbours
    go = base + spread * rnd(N, 1) * rnd(1, D)
    gi = base + spread * rnd(M, 1) * rnd(1, D)
    gi[:: 3] = go[torch.arange(0, M, 3, device=DEV) % N]
    eps = sigma * rnd(N, D)
    log_ev, eig = _run(P, go, eps, gi.contiguous(), sigma)
    ref = _plain(go + eps, gi, sigma)
    assert float(((log_ev - ref).abs() / (1.0 + ref.abs())).max()) <= 1e-12
    e = (-(eps ** 2).sum(-1) / (2 * sigma ** 2) - ref).mean()
    scale = 1.0 + float((eps ** 2).sum(-1).max()) / (2 * sigma ** 2) + float(ref.abs().max())
    assert abs(float(eig.item()) - float(e)) <= 1e-12 * scale
    # the same data one double off a 16-byte boundary
    buf = torch.empty(M * D + 1, dtype=torch.float64, device=DEV)
    buf[1:] = gi.flatten()
    again, _ = _run(P, go, eps, buf[1:].view(M, D), sigma)
    assert torch.equal(again, log_ev)


def test_screened_non_finite(P):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    go = torch.randn((6, 10), dtype=torch.float64, device=DEV, generator=gen)
    gi = torch.randn((300, 10), dtype=torch.float64, device=DEV, generator=gen)
    eps = 0.1 * torch.randn((6, 10), dtype=torch.float64, device=DEV, generator=gen)
    go[2, 3] = float("nan")
    far = gi.clone()
    far[[0, 17, 299]] = float("inf")
    log_ev, _ = _run(P, go, eps, far, 0.5)
    fin = torch.isfinite(far).all(1)
    ref = _plain(go + eps, far[fin], 0.5) + math.log(int(fin.sum()) / 300)
    assert float(log_ev[2]) == -math.inf
    keep = [0, 1, 3, 4, 5]
    assert float((log_ev[keep] - ref[keep]).abs().max()) <= 1e-12 * float(ref[keep].abs().max())
    gi[44, 1] = float("nan")
    log_ev, _ = _run(P, go, eps, gi, 0.5)
    assert bool(torch.isnan(log_ev[keep]).all())
