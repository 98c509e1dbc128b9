"""log-determinants and their sums: matrices in any units (diagonals from 1e-300 to 1e300),
every subset size, matrices that are not positive definite, more nodes than one block, and
per-design sums from records on and off 32-byte boundaries.  The reference is numpy's LU
determinant of the diagonally scaled matrix plus the diagonal's logarithms; an elimination's
error is a few condition numbers of the scaled matrix times 2^-53, here below 1e-12 of the
log-determinant's largest term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LO, HI = [0.0] * 7, [1.0, 2.0, 0.5, 4.0, 1e3, 1e-3, 7.0]


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1502_07873_gb300 as P
    return P


def _spd(n, seed, scale):
    rng = np.random.default_rng(seed)
    J = rng.standard_normal((n, 20, 7))
    H = np.einsum("nij,nik->njk", J, J)
    s = 10.0 ** rng.uniform(-scale, scale, (n, 7))
    return H, s


def _gain(H, s, F):
    """D_KL-hat over F of diag(s) H diag(s)."""
    k = len(F)
    Hf = H[:, F][:, :, F]
    d = np.sqrt(np.einsum("nii->ni", Hf))
    sign, ld = np.linalg.slogdet(Hf / d[:, :, None] / d[:, None, :])
    assert np.all(sign > 0)
    ld = ld + 2 * np.log(d).sum(1) + 2 * np.log(s[:, F]).sum(1)
    return 0.5 * ld - 0.5 * k * (np.log(2 * np.pi) + 1) + np.sum(np.log(np.array(HI)[F] - np.array(LO)[F]))


@pytest.mark.parametrize("n,scale", [(1, 0.0), (511, 10.0), (513, 1.0), (5000, 15.0), (64, 70.0), (64, 150.0)])
def test_gains_in_any_units(P, n, scale):
    H, s = _spd(n, n, scale)
    Hs = H * s[:, :, None] * s[:, None, :]
    ok = np.isfinite(Hs).all((1, 2)) & (np.einsum("nii->ni", Hs) > 0).all(1) if scale > 100 else np.ones(n, bool)
    w = np.random.default_rng(1).uniform(-0.5, 1.0, n)
    for F in ([0], [3, 6], [1, 3, 4], [0, 1, 2, 6], [0, 2, 3, 4, 5], [1, 2, 3, 4, 5, 6], list(range(7))):
        eig = torch.zeros(1, dtype=torch.float64, device=DEV)
        dkl = torch.zeros(n, dtype=torch.float64, device=DEV)
        st = torch.zeros(n, dtype=torch.int32, device=DEV)
        nb = torch.zeros(1, dtype=torch.int32, device=DEV)
        P.oed_eig_subset(None, torch.tensor(Hs, device=DEV), torch.tensor(w, device=DEV), LO, HI, F, eig, dkl=dkl,
                         status=st, n_bad=nb)
        ref = _gain(H, s, F)
        got = dkl.cpu().numpy()
        big = 1.0 + np.abs(np.log(s[:, F])).max(1) * 2 * len(F)
        assert np.all(st.cpu().numpy()[ok] == 0)
        assert np.max(np.abs(got - ref)[ok] / big[ok]) <= 1e-12
        if ok.all():
            assert int(nb.item()) == 0
            assert abs(float(eig.item()) - float(w @ ref)) <= 1e-12 * float(np.abs(w) @ (np.abs(ref) + big))


def test_refused_matrices(P):
    H, _ = _spd(9, 3, 0.0)
    H[1, 2, 2] = 0.0
    H[2, 4, 4] = -1.0
    H[3, 0, 5] = H[3, 5, 0] = np.nan
    H[4, 6, 6] = np.inf
    H[5, :, 3] = H[5, :, 2]          # two equal parameters: singular
    H[5, 3, :] = H[5, 2, :]
    H[5, 3, 3] = H[5, 2, 2]
    H[6] -= 2.0 * np.trace(H[6]) * np.outer(np.ones(7), np.ones(7)) * (1 - np.eye(7))   # indefinite
    H[7] = 0.0
    eig = torch.zeros(1, dtype=torch.float64, device=DEV)
    st = torch.zeros(9, dtype=torch.int32, device=DEV)
    dkl = torch.full((9,), 5.0, dtype=torch.float64, device=DEV)
    nb = torch.zeros(1, dtype=torch.int32, device=DEV)
    P.oed_eig(None, torch.tensor(H, device=DEV), torch.ones(9, dtype=torch.float64, device=DEV), LO, HI, eig, dkl=dkl,
              status=st, n_bad=nb)
    assert st.cpu().tolist() == [0] + [P.OED_ENOTPD] * 7 + [0]
    assert int(nb.item()) == 7 and dkl.cpu().tolist()[1:8] == [0.0] * 7
    assert abs(float(eig.item()) - float(dkl[0] + dkl[8])) == 0.0


@pytest.mark.parametrize("n,nrec,nwin,win", [(1, 1, 1, 0), (257, 5, 3, 1), (40, 91, 2, 1)])
def test_designs_on_any_boundary(P, n, nrec, nwin, win):
    rng = np.random.default_rng(n)
    J = rng.standard_normal((n, nrec, nwin, 9, 7))
    Hr = np.einsum("nrwij,nrwik->nrwjk", J, J).cumsum(2)
    iu = np.triu_indices(7)
    packed = Hr[..., iu[0], iu[1]]
    mask = (rng.random((13, nrec)) < 0.5).astype(np.uint8)
    mask[:, 0] = 1
    w = rng.random(n)
    ref = np.array([w @ _gain(Hr[:, m.astype(bool), win].sum(1), np.ones((n, 7)), list(range(7))) for m in mask])
    out = []
    for off in (0, 1):   # one double off the 32-byte boundary
        buf = torch.zeros(packed.size + off, dtype=torch.float64, device=DEV)
        buf[off:] = torch.tensor(packed.ravel(), device=DEV)
        eig = torch.zeros(13, dtype=torch.float64, device=DEV)
        P.oed_eig_designs(None, buf[off:].view(n, nrec, nwin, 28), win, torch.tensor(mask, device=DEV),
                          torch.tensor(w, device=DEV), LO, HI, eig)
        out.append(eig.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    assert np.max(np.abs(out[0] - ref)) <= 1e-12 * np.max(np.abs(ref)) * 7
