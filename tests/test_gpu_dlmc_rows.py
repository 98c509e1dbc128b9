"""The double loop with more outer samples than one launch's rows: groups of rows whose tiles
would exceed 65535 in a grid's second dimension where there are few inner samples.  Against the
plain FP64 formula to 1e-12 (a handful of FP64 operations a value)."""
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


@pytest.mark.parametrize("N,M,D", [
    (4194240, 3, 2), (4194304, 1, 1), (4793491, 7, 1), (9000001, 2, 3), (4194241, 8, 1),
])
def test_many_outer_few_inner_samples(P, N, M, D):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N)
    go, eps, gi = (torch.randn((k, D), dtype=torch.float64, device=DEV, generator=gen) for k in (N, N, M))
    sigma = 0.4
    log_ev = torch.zeros(N, dtype=torch.float64, device=DEV)
    eig = torch.zeros(1, dtype=torch.float64, device=DEV)
    P.oed_dlmc(go, eps, gi, sigma, log_ev, eig)
    torch.cuda.synchronize()
    l = torch.stack([((go + eps - gi[m]) ** 2).sum(-1) for m in range(M)], 1) / (-2 * sigma ** 2)
    ref = torch.logsumexp(l, 1) - math.log(M)
    assert float(((log_ev - ref).abs() / (1.0 + ref.abs())).max()) <= 1e-12
    e = float((-(eps ** 2).sum(-1) / (2 * sigma ** 2) - ref).mean())
    assert abs(float(eig) - e) <= 1e-10 * (1.0 + abs(e))
