"""Local eigensolves whose subdomains are spread over thread-block clusters, against the oracle."""
import numpy as np
import pytest

from oracle import a2ls_oracle as O
from workloads import pde

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eigp", ["fp64", "fp32x2"])
@pytest.mark.parametrize("m,nb", [(21, 2), (45, 5), (63, 7)])   # clusters of 8, 4 and 2 CTAs
def test_clustered_orthogonalisation_matches_oracle(m, nb, eigp):
    """Row slices of 13 to 60 rows, the last one shorter: the eigenvalues of subdomains that reached the
    target agree with the oracle's to a hundred times the eigen-residual target of 1e-9 (an eigenvalue's error
    is its condition number times the residual), and the selected count is the same."""
    from paper_2201_02250_gb300 import a2ls
    prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=1, nev=4)
    P, _keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, prob.nev, eig_precision=eigp, eig_tol=1e-9)
    ref = O.setup(prob.A, prob.part, prob.overlap, prob.nev)
    ev, res = P.eigenvalues(), P.eig_residuals()
    assert np.sum(res <= 1e-9) >= 0.9 * len(res)
    for i, e in enumerate(ref.eig):
        if res[i] > 1e-9:
            continue
        mine = ev[i][np.isfinite(ev[i].real)]
        # the leading one alone is free of the question which member of a close pair the cut keeps
        assert abs(np.abs(mine).max() - np.abs(e.selected).max()) <= 1e-7 * np.abs(e.selected).max()
    r = np.random.default_rng(1).uniform(-1, 1, prob.n)
    import torch
    b = torch.as_tensor(r, device="cuda")
    x = torch.zeros_like(b)
    it, rr, ok = P.solve(b, x, 1e-8)
    want = O.gmres(prob.A, lambda v: O.apply(ref, v), r, rtol=1e-8)
    assert ok and abs(it - want.iters) <= 1


@pytest.mark.parametrize("eigp", ["fp64", "fp32x2"])
@pytest.mark.parametrize("m,nb", [(47, 2), (83, 5), (112, 7)])   # clusters of 8, 4 and 2 CTAs (FP64: 8, 8 and 4)
def test_clustered_factorisation_matches_oracle(m, nb, eigp):
    """Subdomains of 300 to 650 rows, whose 5 to 11 ragged tiles a block column are dealt to the CTAs of a cluster:
    the quantities and the bounds of the test above, which the factors of both matrices enter."""
    test_clustered_orthogonalisation_matches_oracle(m, nb, eigp)


@pytest.mark.parametrize("m,nb", [(21, 2), (40, 9), (70, 13)])   # 4, 81 and 169 subdomains of 8 columns: chunks of 2, 4 and 8
def test_double_float_chunk_widths_match_oracle(m, nb):
    """The triangular solves without tensor cores at each width of their column chunks: eigenvalues as above."""
    from paper_2201_02250_gb300 import a2ls
    prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=1, nev=4)
    P, _keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, prob.nev, eig_precision="fp32x2", eig_tol=1e-9,
                               tensor_cores=0)
    ref = O.setup(prob.A, prob.part, prob.overlap, prob.nev)
    ev, res = P.eigenvalues(), P.eig_residuals()
    assert np.sum(res <= 1e-9) >= 0.9 * len(res)
    for i, e in enumerate(ref.eig):
        mine = ev[i][np.isfinite(ev[i].real)]
        if res[i] <= 1e-9:
            assert abs(np.abs(mine).max() - np.abs(e.selected).max()) <= 1e-7 * np.abs(e.selected).max()
