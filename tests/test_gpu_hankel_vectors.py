"""The singular triplets that the extraction takes from the Hankel SVD (those above the rank threshold), where most
columns are rounding noise that the Jacobi sweeps orthogonalise only in part.

U and W must be orthonormal up to Jacobi's stop, n eps a pair. H W - U Sigma of a column is what the noise columns keep
of it together: at most the QR's truncation, 1e-14 sigma_1, and the rounding of a QR and Jacobi of order n (u sqrt(n k)
after k <= n steps; n u covers it). So are the singular values.
"""
import ctypes

import numpy as np
import pytest

import synth
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def bnd():
    from paper_1910_11712_gb300 import binding
    binding.load(build_if_missing=True)
    return binding


def _matrix(torch, plan, name, n):
    ptr, nbytes = plan.buffer(name)
    assert nbytes == 16 * n * n
    out = torch.empty(2 * n * n, dtype=torch.float64, device="cuda")
    cudart = ctypes.CDLL("libcudart.so")
    assert cudart.cudaMemcpy(ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(ptr), ctypes.c_size_t(nbytes), 3) == 0
    return out.cpu().numpy().view(np.complex128).reshape(n, n).T


@pytest.mark.parametrize("family,s,L,M", [("drude", 13, 32, 8), ("drude", 24, 16, 8), ("drude", 31, 17, 15),
                                          ("delay", 32, 16, 8), ("sqrt", 7, 24, 8)])
@pytest.mark.parametrize("precision", [0, 1])
def test_triplets_above_the_rank_threshold(bnd, family, s, L, M, precision):
    torch = torch_cuda()
    p = {"drude": synth.drude_2d, "delay": synth.delay_2d, "sqrt": synth.sqrt_3d}[family](s=s, seed=4)
    V = synth.random_probe_block(p.n, L, 3)
    split = bnd.Split.from_problem(p)
    plan = bnd.Plan(split, p.region, 64, L, M, precision=precision)
    plan.execute(torch.from_numpy(np.asfortranarray(V).ravel(order="F").view(np.float64).copy()).cuda())
    res = plan.result()
    n, m = L * M, res["m"]
    H, U, W = (_matrix(torch, plan, k, n) for k in ("H", "U", "W"))
    U, W, sigma = U[:, :m], W[:, :m], res["sigma"]
    assert 0 < m < n
    assert np.abs(U.conj().T @ U - np.eye(m)).max() <= 4 * n * EPS
    assert np.abs(W.conj().T @ W - np.eye(m)).max() <= 4 * n * EPS
    tol = (1e-14 + n * EPS / 2) * sigma[0]
    rest = H.astype(np.clongdouble) @ W - U.astype(np.clongdouble) * sigma[:m]
    assert np.linalg.norm(rest.astype(np.complex128), axis=0).max() <= tol
    assert np.abs(sigma - np.linalg.svd(H, compute_uv=False)).max() <= tol
