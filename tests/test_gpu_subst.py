"""GPU: the blocked banded substitution against the factors it was given, row interchanges included."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(1, 0, 0), (15, 3, 2), (16, 3, 1), (17, 1, 1), (33, 17, 5), (64, 1, 1), (200, 64, 64), (257, 16, 40),
         (320, 100, 44), (400, 143, 143), (420, 60, 200)]


def _band(rng, n, kl, ku):
    A = np.zeros((n, n), complex)
    for o in range(-min(kl, n - 1), min(ku, n - 1) + 1):
        m = n - abs(o)
        A += np.diag(rng.standard_normal(m) + 1j * rng.standard_normal(m), o)
    return A


@pytest.mark.parametrize("precision,u", [(0, 2.0 ** -53), (1, 2.0 ** -24)])
@pytest.mark.parametrize("n,kl,ku", SIZES)
def test_solves_agree_with_the_factors(n, kl, ku, precision, u):
    """Every column of a solve is bitwise the same for 1, 3, 9 and 40 right-hand sides (every launch shape,
    sweeps included), and its residual is that of a substitution with the computed factors:
    |A x - b| <= c m u (|A| + growth) |x| per row with m = kl + ku + 1 terms; random entries of order 1 and
    partial pivoting keep |L| <= sqrt 2 (complex pivots by 1-norm) and U within the growth seen below."""
    import scipy.sparse as sp
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n + 7 * kl + ku)
    A = _band(rng, n, kl, ku)
    split = nep.Split([sp.csr_matrix(A)], [{"kind": "rational", "num": [1.0], "den": None}])
    npts, dt = 3, (torch.complex64 if precision else torch.complex128)
    F = torch.ones(npts, dtype=torch.complex128, device="cuda")
    ab = torch.empty(npts * n * split.ldab, dtype=dt, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    nep.assemble_band(split, npts, F, precision, ab)
    nep.band_factor(split, npts, precision, ab, ipiv, info)
    assert not info.any()
    b = rng.standard_normal((n, 40)) + 1j * rng.standard_normal((n, 40))
    cols = torch.from_numpy(np.ascontiguousarray(b.T)).to(dt).cuda()  # row = one right-hand side
    first = None
    for L in (1, 3, 9, 40):
        B = cols[:L].repeat(npts, 1).contiguous()
        nep.band_solve(split, npts, precision, ab, ipiv, L, B)
        X = B.view(npts, L, n)
        if first is None:
            first = X[:, 0].clone()
        assert torch.equal(torch.view_as_real(X[:, 0].contiguous()), torch.view_as_real(first))
        assert torch.equal(torch.view_as_real(X[0].contiguous()), torch.view_as_real(X[2].contiguous()))
    x = X[1].cpu().numpy().astype(complex).T
    Ad = A.astype(np.complex64).astype(complex) if precision else A
    bd = b.astype(np.complex64).astype(complex) if precision else b
    kv = min(kl + ku, n - 1)
    U = ab.view(npts, n, split.ldab)[1].abs().max().item()
    r = np.abs(Ad @ x - bd).max(0)
    bound = 16 * (kl + 1) * (kv + 1) * u * np.sqrt(2.0) * U * np.abs(x).max(0)
    assert (r <= bound + 16 * u * np.abs(bd).max(0)).all()
