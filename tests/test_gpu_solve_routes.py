"""GPU: which kernel takes a banded solve, and complex128 solves of many right-hand sides by the register sweeps against
the blocked substitution."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivots", [False, True])
@pytest.mark.parametrize("n,kl,ku,npts,L", [(45, 5, 9, 96, 16), (90, 24, 24, 65, 16), (97, 31, 30, 64, 32), (130, 64, 64, 96, 32),
                                            (200, 96, 96, 96, 17), (300, 128, 128, 160, 17), (300, 60, 200, 96, 32)])
def test_columns_equal_single_solves(n, kl, ku, npts, L, pivots):
    """Both kernels apply the same operations to an element in the same order: a column of a solve of many
    right-hand sides is bitwise the solve of that column at two points alone. Interchanges as far as kl rows occur."""
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
    ab = torch.empty(npts * n * split.ldab, dtype=torch.complex128, device="cuda")
    ipiv = torch.empty(npts * n, dtype=torch.int32, device="cuda")
    info = torch.empty(npts, dtype=torch.int32, device="cuda")
    nep.assemble_band(split, npts, F, 0, ab)
    nep.band_factor(split, npts, 0, ab, ipiv, info)
    assert not info.any()
    assert nep.band_solve_kernel(split, npts, 0, L) == "band_sweep_kernel"
    assert nep.band_solve_kernel(split, 2, 0, L) == "band_subst_kernel"
    g = torch.Generator(device="cuda").manual_seed(n)
    B0 = torch.randn((npts, L, n), dtype=torch.complex128, device="cuda", generator=g)
    B = B0.clone()
    nep.band_solve(split, npts, 0, ab, ipiv, L, B)
    for p in (0, npts - 2):
        two = B0[p:p + 2].contiguous()
        nep.band_solve(split, 2, 0, ab.view(npts, -1)[p:p + 2].contiguous(), ipiv.view(npts, n)[p:p + 2].contiguous(), L, two)
        assert torch.equal(torch.view_as_real(B[p:p + 2].contiguous()), torch.view_as_real(two))


def test_batched_plans_equal_single_plans():
    """Plans in plain FP64 whose solves take the sweeps, in shared launches with one whose solves do not."""
    import torch
    import synth
    from paper_1910_11712_gb300 import binding as nep

    plans, V, keep = [], [], []
    for s, N, L in ((24, 96, 16), (20, 128, 32), (12, 32, 8)):
        p = synth.drude_2d(s=s, seed=4)
        split = nep.Split.from_problem(p)
        keep.append(split)
        plans.append(nep.Plan(split, p.region, N, L, 4, precision=nep.NEP_PREC_FP64))
        v = synth.random_probe_block(p.n, L, 3)
        V.append(torch.from_numpy(np.asfortranarray(v).ravel(order="F").view(np.float64).copy()).cuda())
        assert nep.band_solve_kernel(split, N, 0, L) == ("band_sweep_kernel" if s > 12 else "band_subst_kernel")
    alone = []
    for p, v in zip(plans, V):
        p.execute(v)
        alone.append(p.result())
    nep.execute_batch(plans, V)
    for p, a in zip(plans, alone):
        r = p.result()
        assert all(np.array_equal(r[k], a[k]) for k in ("lam", "X", "sigma"))


def test_names_of_the_solve_kernels():
    import scipy.sparse as sp
    from paper_1910_11712_gb300 import binding as nep

    def name(n, k, npts, precision, L):
        A = sp.diags([np.ones(n - abs(o)) * (4.0 if o == 0 else 1.0) for o in (-k, 0, k)], (-k, 0, k), format="csr")
        return nep.band_solve_kernel(nep.Split([A], [{"kind": "rational", "num": [1.0], "den": None}]), npts, precision, L)

    assert name(300, 64, 64, 1, 16) == "band_subst_kernel" and name(300, 64, 128, 1, 32) == "band_sweep_kernel"
    assert name(300, 64, 64, 0, 16) == "band_subst_kernel" and name(1300, 576, 64, 1, 24) == "band_solve_blocked_kernel"
    assert name(1300, 576, 64, 0, 24) == "band_solve_kernel"
