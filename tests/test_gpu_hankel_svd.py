"""The Hankel SVD of a plan (QR with column pivoting, then Jacobi with the pairs of each sweep screened where most
columns are rounding noise) against LAPACK on the plan's own Hankel matrix.

Shapes: both kernels' edges (order 256 is the screened kernel's largest, 257 and up take the full sweeps; odd
orders leave one column without a partner; one block row), few and many significant values. A singular value may
move by the QR's truncation (1e-14 sigma_1) and by FP64 rounding of an SVD of order n (a few n eps sigma_1).
"""
import ctypes

import numpy as np
import pytest

import synth
from oracle import ciss
from tests.gpu_util import match_eigenvalues, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bnd():
    from paper_1910_11712_gb300 import binding
    binding.load(build_if_missing=True)
    return binding


def _hankel(torch, plan, n):
    ptr, nbytes = plan.buffer("H")
    assert nbytes == 16 * n * n
    out = torch.empty(2 * n * n, dtype=torch.float64, device="cuda")
    cudart = ctypes.CDLL("libcudart.so")
    assert cudart.cudaMemcpy(ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(ptr), ctypes.c_size_t(nbytes), 3) == 0
    return out.cpu().numpy().view(np.complex128).reshape(n, n).T


@pytest.mark.parametrize("L,M", [(32, 8), (15, 17), (16, 8), (31, 7), (3, 3), (33, 8), (8, 1)])
@pytest.mark.parametrize("precision", [0, 1])
def test_hankel_singular_values(bnd, L, M, precision):
    torch = torch_cuda()
    p = synth.drude_2d(s=13, seed=4)
    V = synth.random_probe_block(p.n, L, 3)
    split = bnd.Split.from_problem(p)
    plan = bnd.Plan(split, p.region, 64, L, M, precision=precision)
    Vd = torch.from_numpy(np.asfortranarray(V).ravel(order="F").view(np.float64).copy()).cuda()
    plan.execute(Vd)
    res = plan.result()
    n = L * M
    ref = np.linalg.svd(_hankel(torch, plan, n), compute_uv=False)
    tol = (1e-14 + 4 * n * np.finfo(float).eps) * ref[0]
    assert np.abs(res["sigma"] - ref).max() <= tol
    # the values above the rank threshold keep their accuracy relative to sigma_1 / sigma_i
    assert res["m"] == int((ref > 1e-12 * ref[0]).sum()) or np.abs(ref / ref[0] - 1e-12).min() <= 1e-13
    if n > 2 * res["m"]:  # not saturated: the eigenpairs inside
        ora = ciss.solve(p, N=64, L=L, M=M, V=V)
        err, _ = match_eigenvalues(res["lam"], ora["lam"])
        assert err <= 1e-9 and res["eta"].max() <= 1e-10
    plan2 = bnd.Plan(split, p.region, 64, L, M, precision=precision)
    plan2.execute(Vd)
    assert np.array_equal(plan2.result()["sigma"], res["sigma"])  # no dependence on timing
