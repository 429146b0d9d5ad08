"""Matrices with entries that are not finite are refused by the step that has always refused them."""
import numpy as np
import pytest

from workloads import pde

pytestmark = pytest.mark.gpu


def _setup_error(value, entry, **opts):
    """The error code of a set-up whose matrix holds `value` inside the first subdomain (253 rows, four blocks of
    the factorisation)."""
    from paper_2201_02250_gb300 import a2ls
    prob = pde.tiny_conv_diff(m=40, nb=3, overlap=2, nev=6)
    A = prob.A.tocsr().copy()
    row = 5 * 40 + 5
    cols = A.indices[A.indptr[row]:A.indptr[row + 1]]
    A.data[A.indptr[row] + np.flatnonzero((cols == row) == (entry == "diagonal"))[0]] = value
    with pytest.raises(a2ls.A2lsError) as e:
        a2ls.from_scipy(A, prob.part, prob.overlap, prob.nev, **opts)
    return e.value.code


@pytest.mark.parametrize("entry,value", [("diagonal", np.nan), ("off", np.nan), ("off", np.inf), ("off", 1e39)])
def test_tensor_core_digits_keep_what_is_not_finite(entry, value):
    """Static pivoting lets the factorisation pass; the eigensolve's finiteness test sees the products of the
    digits (1e39 is infinite in double-float)."""
    from paper_2201_02250_gb300 import a2ls
    assert _setup_error(value, entry, precision="fp32", tensor_cores=1, static_pivoting=1) == a2ls.A2LS_ERR_EIGEN


@pytest.mark.parametrize("tensor_cores", [0, 1])
@pytest.mark.parametrize("entry", ["diagonal", "off"])
def test_nan_pivot_is_not_a_tiny_one(entry, tensor_cores):
    """A NaN is no small pivot, which would be reported as singular (or replaced): the eigensolve reports it."""
    from paper_2201_02250_gb300 import a2ls
    assert _setup_error(np.nan, entry, precision="fp32", tensor_cores=tensor_cores) == a2ls.A2LS_ERR_EIGEN
