"""The double loop's scratch: what the library keeps of it between calls is bounded (256 MB), is given
back when a context is destroyed, and is shared by threads with streams of their own without a
bit of the results changing."""
import threading

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MB = 1 << 20


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1502_07873_gb300 as P
    return P


def _data(N, M, D):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N + M + D)
    go, gi, eps = (torch.randn((k, D), dtype=torch.float64, device=DEV, generator=gen) for k in (N, M, N))
    out = torch.zeros(N, dtype=torch.float64, device=DEV), torch.zeros(1, dtype=torch.float64, device=DEV)
    return go, 0.3 * eps, gi, 0.3, *out


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_scratch_is_bounded_and_given_back(P):
    small, large = _data(300, 200, 20), _data(9000, 6000, 3000)   # large: 180 MB of data, 128 MB of distances
    P.oed_dlmc(*small)
    ctx = P.Context(P.problem_from_workload(W.tiny(), P.OED_FP32), max_solves=1)   # (and loads the kernels)
    ctx.close()
    before = _free()
    for _ in range(3):
        P.oed_dlmc(*large)
        P.oed_dlmc(*small)
        assert before - _free() <= 260 * MB
    ctx = P.Context(P.problem_from_workload(W.tiny(), P.OED_FP32), max_solves=1)
    ctx.close()
    assert before - _free() <= 4 * MB


def test_threads_and_streams(P):
    sizes = [(300, 200, 20), (2000, 1500, 60), (700, 3000, 33), (65, 129, 31)]
    ref = []
    for s in sizes:
        d = _data(*s)
        P.oed_dlmc(*d)
        torch.cuda.synchronize()
        ref.append((d[4].clone(), d[5].clone()))
    bad = []

    def work(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for i in range(12):
                q = (k + i) % len(sizes)
                d = _data(*sizes[q])
                P.oed_dlmc(*d, stream=stream)
                stream.synchronize()
                if not (torch.equal(d[4], ref[q][0]) and torch.equal(d[5], ref[q][1])):
                    bad.append((k, i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_captured(P):
    go, eps, gi, sigma, log_ev, eig = _data(500, 400, 50)
    P.oed_dlmc(go, eps, gi, sigma, log_ev, eig)
    torch.cuda.synchronize()
    ref = log_ev.clone(), eig.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.oed_dlmc(go, eps, gi, sigma, log_ev, eig)
    for _ in range(2):
        log_ev.zero_()
        eig.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(log_ev, ref[0]) and torch.equal(eig, ref[1])
