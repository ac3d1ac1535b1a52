"""The widest complex64 bands around the limit of the tensor-core LU's shared memory (kl = 854; the panel of a wider
band does not fit beside the kernel's static part) factor and solve on either side of it, with a normwise backward
error within the first-order bound of FP32 elimination."""
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


@pytest.mark.parametrize("kl", [701, 853, 854, 855, 856, 857, 870])
@pytest.mark.parametrize("npts", [1, 80])
def test_widest_bands(bnd, kl, npts):
    torch = torch_cuda()
    n, ku = 1000, 5
    rng = np.random.default_rng(kl)
    offs = list(range(-kl, ku + 1))
    A = sp.diags([rng.standard_normal(n - abs(o)) + 1j * rng.standard_normal(n - abs(o)) for o in offs], offs, format="csr")
    split = bnd.Split([A], [{"kind": "rational", "num": [1.0], "den": None}])
    F = torch.ones(npts, dtype=torch.complex128, device="cuda")
    ab = torch.empty(npts * n * split.ldab, dtype=torch.complex64, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    bnd.assemble_band(split, npts, F, 1, ab)
    bnd.band_factor(split, npts, 1, ab, ipiv, info)
    assert int(info.abs().sum()) == 0
    b = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
    B = torch.from_numpy(np.tile(b, npts)).cuda()
    bnd.band_solve(split, npts, 1, ab, ipiv, 1, B)
    X = B.cpu().numpy().reshape(npts, n).astype(np.complex128)
    scale = abs(A).sum(axis=1).max()
    for x in (X[0], X[-1]):
        r = np.abs(A @ x - b).max() / (scale * np.abs(x).max() + np.abs(b).max())
        assert r <= (2 * kl + ku) * np.finfo(np.float32).eps
