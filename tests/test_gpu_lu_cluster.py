"""The tensor-core banded LU on two CTAs per point (few points) and on one (many points): the same factors bit for
bit, and a normwise backward error of the solves within the first-order bound of FP32 elimination.

Bands at the panel's edges: 97 rows (three groups of 32 and one row more), 512 and 513 rows (one and two groups a
warp), and the widest panel with the scratch beside it; n around multiples of 32; bands with many interchanges.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bnd():
    from paper_1910_11712_gb300 import binding
    binding.load(build_if_missing=True)
    return binding


def _band(n, kl, ku, seed):
    rng = np.random.default_rng(seed)
    offs = list(range(-kl, ku + 1))
    return sp.diags([rng.standard_normal(n - abs(o)) + 1j * rng.standard_normal(n - abs(o)) for o in offs], offs,
                    format="csr")


@pytest.mark.parametrize("n,kl,ku", [(200, 65, 65), (131, 66, 3), (192, 66, 100), (1000, 480, 20), (1001, 481, 20),
                                     (1500, 700, 40)])
def test_two_ctas_per_point_match_one(bnd, n, kl, ku):
    torch = torch_cuda()
    A = _band(n, kl, ku, n + kl)
    split = bnd.Split([A], [{"kind": "rational", "num": [1.0], "den": None}])
    out = []
    for npts in (2, 80):  # 80 points: one CTA each (two would not be resident at once)
        F = torch.ones(npts, dtype=torch.complex128, device="cuda")
        ab = torch.empty(npts * n * split.ldab, dtype=torch.complex64, device="cuda")
        ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
        info = torch.empty(npts, dtype=torch.int32, device="cuda")
        bnd.assemble_band(split, npts, F, 1, ab)
        bnd.band_factor(split, npts, 1, ab, ipiv, info)
        assert int(info.abs().sum()) == 0
        out.append((torch.view_as_real(ab).view(npts, -1)[:2].clone(), ipiv.view(npts, n)[:2].clone()))
        if npts == 2:
            rng = np.random.default_rng(1)
            b = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
            B = torch.from_numpy(np.tile(b, 2)).cuda()
            bnd.band_solve(split, 2, 1, ab, ipiv, 1, B)
            x = B.cpu().numpy()[:n].astype(np.complex128)
            r = np.abs(A @ x - b).max() / (abs(A).sum(axis=1).max() * np.abs(x).max() + np.abs(b).max())
            assert r <= (2 * kl + ku) * np.finfo(np.float32).eps
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
