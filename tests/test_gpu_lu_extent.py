"""GPU: factorisations and solves that stop at the columns the interchanges so far can reach."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# register window (kl <= 64), tensor-core and blocked kernels; sizes off the 16, 32, 64 and 128 tiles
SIZES = [(40, 3, 0), (90, 1, 30), (150, 20, 12), (301, 33, 31), (400, 64, 64), (420, 66, 1), (500, 97, 97), (610, 100, 150),
         (1000, 290, 150)]


def _matrix(rng, n, kl, ku, pivots):
    A = np.zeros((n, n), complex)
    for o in range(-kl, ku + 1):
        m = n - abs(o)
        A += np.diag(rng.standard_normal(m) + 1j * rng.standard_normal(m), o)
    if pivots != "all":  # the diagonal stays the largest of its column
        A[np.arange(n), np.arange(n)] = 4.0 * (kl + ku + 1)
    if pivots == "few":  # rows n/3 and 2n/3 trade places with rows kl and kl/2 + 1 below
        for c, d in ((n // 3, kl), (2 * n // 3, kl // 2 + 1)):
            d = min(d, kl)
            A[c, c], A[c + d, c] = 1e-3, 4.0 * (kl + ku + 1)
    return A


@pytest.mark.parametrize("pivots", ["none", "few", "all"])
@pytest.mark.parametrize("precision,u", [(0, 2.0 ** -53), (1, 2.0 ** -24)])
@pytest.mark.parametrize("n,kl,ku", SIZES)
def test_factor_and_solve(n, kl, ku, precision, u, pivots):
    """A x = b by the computed factors. A residual element sums the roundings of up to (kl+1)(kl+ku+1) products
    l u x, each at most u |l| |u| |x| with |l| <= sqrt 2: taken as independent, their sum stays below 16 standard
    deviations; the split TF32 products of wide complex64 bands round at 4 u."""
    import scipy.sparse as sp
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n + 31 * kl + ku)
    A = _matrix(rng, n, kl, ku, pivots)
    if precision:
        A = A.astype(np.complex64).astype(complex)
    split = nep.Split([sp.csr_matrix(A)], [{"kind": "rational", "num": [1.0], "den": None}])
    npts, L, dt = 2, 17, (torch.complex64 if precision else torch.complex128)
    F = torch.ones(npts, dtype=torch.complex128, device="cuda")
    ab = torch.empty(npts * n * split.ldab, dtype=dt, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    nep.assemble_band(split, npts, F, precision, ab)
    nep.band_factor(split, npts, precision, ab, ipiv, info)
    assert not info.any()
    moved = (ipiv.view(npts, n).cpu().numpy() != np.arange(n)).sum(1)
    assert moved[0] == moved[1] and (moved[0] == 0 if pivots == "none" else moved[0] >= 2)
    b = (rng.standard_normal((n, L)) + 1j * rng.standard_normal((n, L))).astype(np.complex64).astype(complex)
    B = torch.from_numpy(np.ascontiguousarray(b.T)).to(dt).cuda().repeat(npts, 1).contiguous()
    nep.band_solve(split, npts, precision, ab, ipiv, L, B)
    top = ab.abs().max().item()
    unit = 4 * u if precision and kl > 64 else u
    for x in B.view(npts, L, n).cpu().numpy().astype(complex):
        r = np.abs(A @ x.T - b).max(0)
        assert (r <= 16 * unit * np.sqrt(2.0 * (kl + 1) * (kl + ku + 1)) * top * np.abs(x).max(1)).all()
