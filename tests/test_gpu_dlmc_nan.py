"""Not-a-number distances of the double loop.  Where a row of outer data has a distance that
can be compared, one inner sample that is NaN makes its log-evidence NaN, wherever the sample
stands among the others and however many there are: alone in its warp, alone in the last round
of a block, first or last.  The estimate is NaN with it.  A row with no comparable distance (one NaN inner sample)
gives -inf."""
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


def _run(P, M, at, D=12, N=3):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M)
    go, eps, gi = (torch.randn((k, D), dtype=torch.float64, device=DEV, generator=gen) for k in (N, N, M))
    gi[at, D // 2] = float("nan")
    log_ev = torch.zeros(N, dtype=torch.float64, device=DEV)
    eig = torch.zeros(1, dtype=torch.float64, device=DEV)
    P.oed_dlmc(go, 0.1 * eps, gi, 0.5, log_ev, eig)
    torch.cuda.synchronize()
    return log_ev, eig


@pytest.mark.parametrize("M,at", [
    (2, 0), (2, 1), (32, 31), (33, 32), (33, 0), (64, 40), (65, 64), (97, 96), (128, 127), (129, 128), (257, 256),
    (300, 299), (1025, 1024), (2049, 2048), (2049, 100), (5000, 4999),
])
@pytest.mark.parametrize("D", [12, 12290])   # the row's data in shared memory, and not
def test_one_nan_sample_is_seen(P, M, at, D):
    log_ev, eig = _run(P, M, at, D)
    assert bool(torch.isnan(log_ev).all()) and math.isnan(float(eig)), (log_ev, eig)


def test_no_comparable_sample(P):
    log_ev, _ = _run(P, 1, 0)
    assert log_ev.tolist() == [-math.inf] * 3
