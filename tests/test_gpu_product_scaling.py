"""FP64 products of operands that are scaled unevenly, against extended-precision sums, element by element.

An inner product of n complex terms in FP64 has an error of at most about n eps sum |a||b| however its terms are
scaled. Terms of opposite scale (a small where b is large) and entries far below the largest of their row or column
are where products formed from a fixed number of digits below that largest entry would not keep it.
"""
import numpy as np
import pytest

from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def bnd():
    from paper_1910_11712_gb300 import binding
    binding.load(build_if_missing=True)
    return binding


def _dev(torch, a):
    a = np.asarray(a, dtype=np.complex128)
    return torch.from_numpy(np.ascontiguousarray(a.ravel(order="F")).view(np.float64).copy()).cuda()


def _cplx(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _scales(rng, n, s):
    """1/s, s or 1 for every term, each of them at least once where there is room."""
    e = rng.integers(-1, 2, n)
    e[: min(n, 3)] = [-1, 1, 0][: min(n, 3)]
    return float(s) ** rng.permutation(e)


@pytest.mark.parametrize("n,P,nv", [(2, 1, 1), (16, 2, 3), (64, 33, 8), (65, 8, 9), (300, 70, 5)])
@pytest.mark.parametrize("s", [1e3, 1e6, 1e10, 1e60])
def test_dense_products(bnd, n, P, nv, s):
    """D = Y^H V with V scaled by d and Y by 1 / d, then X (D / (z - lambda)) with the columns of X scaled likewise."""
    torch = torch_cuda()
    rng = np.random.default_rng(n + P)
    lam, X, Y, z, V = _cplx(rng, P), _cplx(rng, n, P), _cplx(rng, n, P), 8 + _cplx(rng, 1), _cplx(rng, n, nv)
    d, e = _scales(rng, n, s), _scales(rng, P, s)
    V, Y, X = V * d[:, None], Y / d[:, None] * e, X / e
    out = torch.empty(2 * n * nv, dtype=torch.float64, device="cuda")
    args = [_dev(torch, a) for a in (lam, X, Y, z, V)]
    bnd.apply_resolvent(n, P, args[0], args[1], args[2], 1, args[3], nv, args[4], out)
    got = out.cpu().numpy().view(np.complex128).reshape(nv, n).T
    w = z[0].astype(np.clongdouble) - lam.astype(np.clongdouble)
    ref = X.astype(np.clongdouble) @ ((Y.conj().T.astype(np.clongdouble) @ V.astype(np.clongdouble)) / w[:, None])
    size = np.abs(X) @ ((np.abs(Y).T @ np.abs(V)) / np.abs(w)[:, None])
    # n + P terms, two roundings each per component, and those of the weights
    assert (np.abs(got - ref) <= 4 * (n + P + 4) * EPS * size).all()


@pytest.mark.parametrize("n,L,N,K", [(1, 1, 2, 1), (37, 3, 7, 3), (64, 8, 64, 16), (50, 3, 65, 9), (33, 2, 192, 17)])
@pytest.mark.parametrize("s", [1e3, 1e6, 1e10, 1e60])
def test_moments(bnd, n, L, N, K, s):
    """Coefficients scaled by d over the nodes and Y by 1 / d, each column of Y with its own d."""
    torch = torch_cuda()
    rng = np.random.default_rng(n * N + K)
    nl = n * L
    C, Y = _cplx(rng, K, N), _cplx(rng, N, nl)
    d = _scales(rng, N, s)
    C *= d[None]
    Y[:, ::2] /= d[:, None]
    Y[:, 1::3] *= 10.0 ** rng.uniform(-12, 0, (N, Y[:, 1::3].shape[1]))
    S = torch.empty(K * nl * 2, dtype=torch.float64, device="cuda")
    bnd.moments(n, L, N, K, _dev(torch, C.T), torch.from_numpy(Y.view(np.float64).reshape(-1).copy()).cuda(), S)
    out = S.cpu().numpy().view(np.complex128).reshape(K, nl)
    ref = C.astype(np.clongdouble) @ Y.astype(np.clongdouble)
    assert (np.abs(out - ref) <= 4 * N * EPS * (np.abs(C) @ np.abs(Y))).all()


@pytest.mark.parametrize("zeros", [False, True])
def test_subnormal_columns(bnd, zeros):
    """A column all of whose entries are subnormal is not a zero column; beside exactly zero ones or not."""
    torch = torch_cuda()
    rng = np.random.default_rng(5)
    n, L, N, K = 20, 2, 16, 8
    nl = n * L
    C, Y = _cplx(rng, K, N) * 1e20, _cplx(rng, N, nl)
    Y[:, 3] *= 1e-315
    if zeros:
        Y[:, 4:9] = 0.0
    S = torch.empty(K * nl * 2, dtype=torch.float64, device="cuda")
    bnd.moments(n, L, N, K, _dev(torch, C.T), torch.from_numpy(Y.view(np.float64).reshape(-1).copy()).cuda(), S)
    out = S.cpu().numpy().view(np.complex128).reshape(K, nl)
    ref = C.astype(np.clongdouble) @ Y.astype(np.clongdouble)
    assert (np.abs(out - ref) <= 4 * N * EPS * (np.abs(C) @ np.abs(Y))).all()
    P, nv = 5, 4
    lam, X, Yl, z, V = _cplx(rng, P), _cplx(rng, n, P), _cplx(rng, n, P) * 1e20, 8 + _cplx(rng, 1), _cplx(rng, n, nv)
    V[:, 1] *= 1e-315
    if zeros:
        V[:, 2] = 0.0
    o = torch.empty(2 * n * nv, dtype=torch.float64, device="cuda")
    a = [_dev(torch, v) for v in (lam, X, Yl, z, V)]
    bnd.apply_resolvent(n, P, a[0], a[1], a[2], 1, a[3], nv, a[4], o)
    got = o.cpu().numpy().view(np.complex128).reshape(nv, n).T
    w = (z[0] - lam)[:, None]
    ref = X.astype(np.clongdouble) @ ((Yl.conj().T.astype(np.clongdouble) @ V.astype(np.clongdouble)) / w)
    size = np.abs(X) @ ((np.abs(Yl).T @ np.abs(V)) / np.abs(w))
    assert (np.abs(got - ref) <= 4 * (n + P + 4) * EPS * size).all()
