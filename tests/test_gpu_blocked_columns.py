"""GPU: the blocked substitution of wide complex64 bands at every number of columns per CTA."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivots", [False, True])
@pytest.mark.parametrize("n,kl,ku", [(700, 288, 30), (811, 300, 200), (1300, 577, 577)])
def test_residuals(n, kl, ku, pivots):
    """A x = b by the computed factors with 3, 11, 16 and 33 columns (4, 12, 16 and 12 per CTA). A residual element sums
    the roundings of up to (kl+1)(kl+ku+1) products at most 4 u |l| |u| |x| each (split TF32 products in the
    factorisation), |l| <= sqrt 2: taken as independent, below 16 standard deviations."""
    import scipy.sparse as sp
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n)
    off = range(-kl, ku + 1)
    A = sp.diags([rng.standard_normal(n - abs(o)) + 1j * rng.standard_normal(n - abs(o))
                  + (0 if pivots or o else 4.0 * (kl + ku + 1)) for o in off], list(off), format="csr")
    A = A.astype(np.complex64).astype(complex)
    split = nep.Split([A], [{"kind": "rational", "num": [1.0], "den": None}])
    npts = 2
    F = torch.ones(npts, dtype=torch.complex128, device="cuda")
    ab = torch.empty(npts * n * split.ldab, dtype=torch.complex64, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    nep.assemble_band(split, npts, F, 1, ab)
    nep.band_factor(split, npts, 1, ab, ipiv, info)
    assert not info.any()
    top = ab.abs().max().item()
    bound = 16 * 4 * 2.0 ** -24 * np.sqrt(2.0 * (kl + 1) * (kl + ku + 1)) * top
    for L in (3, 11, 16, 33):
        b = (rng.standard_normal((L, n)) + 1j * rng.standard_normal((L, n))).astype(np.complex64)
        B = torch.from_numpy(b).cuda().repeat(npts, 1).contiguous()
        nep.band_solve(split, npts, 1, ab, ipiv, L, B)
        for x in B.view(npts, L, n).cpu().numpy().astype(complex):
            r = np.abs((A @ x.T).T - b).max(1)
            assert (r <= bound * np.abs(x).max(1)).all()
