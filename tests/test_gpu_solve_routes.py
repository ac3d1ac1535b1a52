"""GPU: which kernel takes a banded solve."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_names_of_the_solve_kernels():
    import scipy.sparse as sp
    from paper_1910_11712_gb300 import binding as nep

    def name(n, k, npts, precision, L):
        A = sp.diags([np.ones(n - abs(o)) * (4.0 if o == 0 else 1.0) for o in (-k, 0, k)], (-k, 0, k), format="csr")
        return nep.band_solve_kernel(nep.Split([A], [{"kind": "rational", "num": [1.0], "den": None}]), npts, precision, L)

    assert name(300, 64, 64, 1, 16) == "band_subst_kernel" and name(300, 64, 128, 1, 32) == "band_sweep_kernel"
    assert name(300, 64, 64, 0, 16) == "band_subst_kernel" and name(1300, 576, 64, 1, 24) == "band_solve_blocked_kernel"
    assert name(1300, 576, 64, 0, 24) == "band_solve_kernel"
