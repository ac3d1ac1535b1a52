"""The FP64 products computed from exact 8-bit digit products (moments, dense products) against extended-precision
sums.

Every result is a sum of exact integers cut at 2^-52 of the largest row and column product at the worst, rounded
once per 64 terms; so the error of a result's norm is at most a few eps (2.2e-16), where plain FP64 FMAs
accumulate one rounding per term. Sizes around the tiles (8 moments, 8 columns, 64 nodes; 32 x 32 tiles,
blocks of 64 terms), values that span many orders of magnitude across nodes, and columns with entries that are not
finite or too large or small for the digits (which take FP64 sums).
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


@pytest.mark.parametrize("n,L,N,K", [(1, 1, 1, 1), (37, 3, 7, 3), (64, 8, 32, 8), (13, 5, 64, 16), (50, 3, 65, 9),
                                     (33, 2, 192, 17), (20, 2, 193, 16)])
@pytest.mark.parametrize("kind", ["normal", "range", "special"])
def test_moments(bnd, n, L, N, K, kind):
    torch = torch_cuda()
    rng = np.random.default_rng(n * N + K)
    nl = n * L
    z = np.cos(2 * np.pi * (np.arange(N) + 0.5) / N) + 0.3j * np.sin(2 * np.pi * (np.arange(N) + 0.5) / N)
    C = (z / N)[None] * z[None] ** np.arange(K)[:, None]
    Y = rng.standard_normal((N, nl)) + 1j * rng.standard_normal((N, nl))
    if kind == "range":
        Y *= 10.0 ** rng.uniform(-4, 4, (N, nl))
    if kind == "special":
        Y[N // 2, 0] = np.inf
        Y[0, nl // 2] = np.nan
        Y[:, nl - 1] *= 1e-200
        Y[0, nl // 3] = 0.0
    S = torch.empty(K * nl * 2, dtype=torch.float64, device="cuda")
    bnd.moments(n, L, N, K, _dev(torch, C.T), torch.from_numpy(Y.view(np.float64).reshape(-1).copy()).cuda(), S)
    out = S.cpu().numpy().view(np.complex128).reshape(K, nl)
    ref = np.zeros((K, nl), np.clongdouble)
    with np.errstate(invalid="ignore"):
        for j in range(N):
            ref += C[:, j].astype(np.clongdouble)[:, None] * Y[j].astype(np.clongdouble)[None]
    good = np.isfinite(ref.astype(np.complex128)).all(axis=0)
    assert np.array_equal(np.isfinite(out).all(axis=0), good)
    d = np.abs(out[:, good] - ref[:, good])
    size = (np.abs(C) @ np.abs(np.where(np.isfinite(Y), Y, 0)))[:, good]
    if kind == "special" or N > 192:  # FP64 FMAs somewhere: one rounding per term and component
        assert (d <= 4 * N * EPS * size).all()
    else:
        assert np.linalg.norm(d.astype(float)) <= (1 + (N + 63) // 64) * EPS * np.linalg.norm(ref.astype(np.complex128))


@pytest.mark.parametrize("n,P,nz,nv", [(1, 1, 1, 1), (64, 8, 1, 32), (65, 33, 2, 5), (301, 31, 3, 11), (1000, 70, 1, 9)])
@pytest.mark.parametrize("special", [0, 1])
def test_dense_products(bnd, n, P, nz, nv, special):
    """nep_apply_resolvent is two dense products: D = Y^H V, then X times (D weighted by 1 / (z - lambda))."""
    torch = torch_cuda()
    rng = np.random.default_rng(n + P)
    c = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    lam, X, Y, z, V = c(P), c(n, P), c(n, P), 8 + c(nz), c(n, nv)
    if special:
        X[0, 0] *= 1e300
        V[n - 1, nv - 1] = 0.0
        Y[n // 2] = 0.0
    out = torch.empty(2 * n * nz * nv, dtype=torch.float64, device="cuda")
    args = [_dev(torch, a) for a in (lam, X, Y, z, V)]
    bnd.apply_resolvent(n, P, args[0], args[1], args[2], nz, args[3], nv, args[4], out)
    got = out.cpu().numpy().view(np.complex128).reshape(nz * nv, n).T
    D = Y.conj().T.astype(np.clongdouble) @ V.astype(np.clongdouble)
    W = np.concatenate([D / (z[j].astype(np.clongdouble) - lam.astype(np.clongdouble))[:, None] for j in range(nz)], 1)
    ref = X.astype(np.clongdouble) @ W
    # rounding of D and of the weights, n and P terms: relative to the sums of moduli
    aW = np.concatenate([(np.abs(Y).T @ np.abs(V)) / np.abs(z[j] - lam)[:, None] for j in range(nz)], 1)
    assert (np.abs(got - ref) <= 8 * (P + n) * EPS * (np.abs(X) @ aW)).all()
    if not special:
        assert np.linalg.norm((got - ref).astype(np.complex128)) <= 16 * EPS * np.linalg.norm(np.abs(X) @ aW)
