"""GPU: register-window sweeps whose window is exactly the bandwidth, against the blocked substitution."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivots", [False, True])
@pytest.mark.parametrize("n,kl,ku", [(70, 32, 32), (70, 32, 5), (130, 64, 64), (131, 40, 64), (200, 96, 96), (300, 128, 128),
                                     (300, 64, 200), (90, 33, 31), (90, 5, 0)])
@pytest.mark.parametrize("npts,L", [(33, 32), (128, 17), (128, 32)])  # one, two and four columns per warp
def test_columns_equal_single_solves(npts, L, n, kl, ku, pivots):
    """Both kernels apply the same operations to an element in the same order: a column of a solve of many
    right-hand sides is bitwise the solve of that column alone. Interchanges as far as kl rows occur."""
    import scipy.sparse as sp
    import torch
    from paper_1910_11712_gb300 import binding as nep

    rng = np.random.default_rng(n + kl + L)
    off = range(-kl, ku + 1)
    A = sp.diags([rng.standard_normal(n - abs(o)) + (0 if pivots or o else 4.0 * (kl + ku + 1)) for o in off], list(off),
                 format="lil", dtype=complex)
    if pivots:
        for c in range(0, n - kl, 7):
            A[c + kl, c] = 50.0  # the farthest row wins the column
    split = nep.Split([A.tocsr()], [{"kind": "rational", "num": [1.0], "den": None}])
    F = torch.from_numpy(1.0 + 0.01 * np.arange(npts) + 0j).cuda()
    ab = torch.empty(npts * n * split.ldab, dtype=torch.complex64, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    nep.assemble_band(split, npts, F, 1, ab)
    nep.band_factor(split, npts, 1, ab, ipiv, info)
    assert not info.any()
    far = (ipiv.view(npts, n).cpu() - torch.arange(n, dtype=torch.int32)).amax().item()
    assert far == (kl if pivots else 0)
    g = torch.Generator(device="cuda").manual_seed(n)
    B0 = torch.randn((npts, L, n), dtype=torch.complex64, device="cuda", generator=g)
    B = B0.clone()
    nep.band_solve(split, npts, 1, ab, ipiv, L, B)
    for l in (0, L // 2, L - 1):
        one = B0[:, l].contiguous()
        nep.band_solve(split, npts, 1, ab, ipiv, 1, one)
        assert torch.equal(torch.view_as_real(B[:, l].contiguous()), torch.view_as_real(one))
