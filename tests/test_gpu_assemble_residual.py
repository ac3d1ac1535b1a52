"""GPU: assembly in groups of rows and residuals of several right-hand sides per thread, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _terms(rng, n, kl, ku, complex_terms, density):
    import scipy.sparse as sp

    out = []
    for _ in range(3):
        d = {o: rng.standard_normal(n - abs(o)) * (rng.random(n - abs(o)) < density)
             for o in range(-min(kl, n - 1), min(ku, n - 1) + 1)}
        A = sp.diags(list(d.values()), list(d), shape=(n, n), format="csr", dtype=complex if complex_terms else float)
        if complex_terms:
            A = A + 1j * A.multiply(rng.standard_normal())
        A.eliminate_zeros()
        out.append(A.tocsr())
    out[0] = (out[0] + sp.eye(n)).tocsr()
    return out


def _split(mats):
    from paper_1910_11712_gb300 import binding as nep

    return nep.Split(mats, [{"kind": "rational", "num": [1.0], "den": None}] * len(mats))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,kl,ku,complex_terms,density",
                         [(1, 0, 0, False, 1.0), (15, 2, 1, True, 1.0), (16, 1, 1, False, 0.4), (17, 3, 0, True, 0.2),
                          (33, 8, 5, False, 1.0), (100, 40, 30, True, 0.9), (259, 16, 16, False, 0.1)])
def test_assembly(n, kl, ku, complex_terms, density, precision):
    """Band entries: three products and sums in FP64, at most 4 u sum |F| |a| each, then one rounding; the norm: sums
    of up to n moduli, (n + 8) u relative."""
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n + kl)
    mats = _terms(rng, n, kl, ku, complex_terms, density)
    split = _split(mats)
    npts, dt = 3, (torch.complex64 if precision else torch.complex128)
    F = rng.standard_normal((3, npts)) + 1j * rng.standard_normal((3, npts))
    ab = torch.full((npts * n * split.ldab + 1,), 7.0, dtype=dt, device="cuda")[1:]  # off the 16-byte boundary
    tnorm = torch.empty(npts, dtype=torch.float64, device="cuda")
    nep.assemble_band(split, npts, torch.from_numpy(np.ascontiguousarray(F.T)).cuda(), precision, ab, tnorm)
    band = ab.view(npts, n, split.ldab).cpu().numpy()
    for j in range(npts):
        T = sum(F[i, j] * mats[i].toarray() for i in range(3))
        size = sum(abs(F[i, j]) * np.abs(mats[i].toarray()) for i in range(3))
        got = np.zeros((n, n), complex)
        rest = band[j].copy()
        for r in range(n):
            for k in range(max(0, r - split.kl), min(n, r + split.ku + 1)):
                got[r, k] = band[j, r, k - r + split.kl]
                rest[r, k - r + split.kl] = 0
        assert not rest.any()
        assert (np.abs(got - T) <= (8 * U + (2.0 ** -23 if precision else 0)) * size).all()
        assert abs(tnorm[j].item() - np.abs(T).sum(1).max()) <= (n + 8) * U * size.sum(1).max()


@pytest.mark.parametrize("n,npts,L", [(1, 2, 4), (300, 152, 4), (300, 152, 5), (513, 102, 7), (300, 3, 9), (256, 700, 1)])
def test_residual(n, npts, L):
    """V - T Y row by row: at most 6 complex products (9 in T's diagonals), each within 8 u |t| |y| with T's own
    rounding, summed in order."""
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n + L)
    mats = _terms(rng, n, 3, 2, True, 0.7)
    split = _split(mats)
    F = rng.standard_normal((3, npts)) + 1j * rng.standard_normal((3, npts))
    V = rng.standard_normal((L, n)) + 1j * rng.standard_normal((L, n))
    Y = rng.standard_normal((npts, L, n)) + 1j * rng.standard_normal((npts, L, n))
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (F.T, V, Y)]
    R = torch.empty((npts, L, n), dtype=torch.complex128, device="cuda")
    nep.split_residual(split, npts, dev[0], L, dev[1], dev[2], R)
    got = R.cpu().numpy()
    for j in range(npts):
        T = sum(F[i, j] * mats[i] for i in range(3))
        size = sum(abs(F[i, j]) * abs(mats[i]) for i in range(3))
        want = V - (T @ Y[j].T).T
        bound = 16 * U * (np.abs(V) + (size @ np.abs(Y[j]).T).T)
        assert (np.abs(got[j] - want) <= bound).all()
