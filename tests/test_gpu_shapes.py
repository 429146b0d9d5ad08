"""Kernels chosen by size, on both sides of the line and at ragged sizes, against scipy and the oracle."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import a2ls_oracle as O
from oracle import gnn_oracle as G
from workloads import pde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [1, 31, 33, 65, 301])   # a thread a row up to 32 entries, a warp above
def test_spmv_by_row_length(width):
    """Rows of 1 .. width entries; the bound is that of any summation order, width 2^-53 |A| |x|, times two."""
    from paper_2201_02250_gb300 import a2ls
    n, r = 1003, np.random.default_rng(width)
    A = sp.lil_matrix((n, n))
    for i in range(n):
        h = min(i, n - 1 - i, (width - 1) // 2)
        A[i, i - h:i + h + 1] = r.uniform(-1, 1, 2 * h + 1) / width
    A = (A + sp.diags(np.full(n, 4.0))).tocsr()
    P, _keep = a2ls.from_scipy(A, (np.arange(n) * 4 // n).astype(np.int32), 1, 1)
    x = r.uniform(-1, 1, n)
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    P.spmv(torch.as_tensor(x, device="cuda"), y)
    bound = 2 * (width + 1) * 2.0**-53 * (abs(A) @ abs(x))
    assert np.all(np.abs(y.cpu().numpy() - A @ x) <= bound)


@pytest.mark.parametrize("m,nb", [
    (142, 2),   # over 5000 rows a subdomain: propagation through global memory; a cluster of 8 for the loss
                # (forward and loss only: FP32 alone moves this size's gradients by 2e-3 to 4e-3)
    (43, 5),    # 25 subdomains, clusters of 4
    (41, 8),    # 64, of 2
    (41, 10),   # 100, one CTA each
])
def test_network_by_subdomain_size_and_count(m, nb):
    """Forward to 1e-4 a subdomain, loss to 1e-4 and gradients to 2e-3 a group: the bounds of the network's
    tests (FP32 accumulation with the same bfloat16 weights)."""
    from paper_2201_02250_gb300 import a2ls
    prob = pde.tiny_conv_diff(m=m, nb=nb, overlap=2, nev=2)
    P, _keep = a2ls.from_scipy(prob.A, prob.part, prob.overlap, prob.nev)
    S = a2ls.GnnSample(P)
    inputs, Z, off = [], [], [0]
    for sub in O.overlapping_subdomains(prob.A, prob.part, prob.overlap):
        lump = np.zeros(sub.n_i)
        lump[sub.n_I:] = O.lumped_row_sums(prob.A, sub)
        inputs.append((O.local_matrix(prob.A, sub), lump, sub.n_I))
        Z.append(np.linalg.qr(np.cos(np.pi * np.outer(np.arange(sub.n_i) + 0.5, 1 + np.arange(1 + len(Z) % 3)) / sub.n_i))[0])
        off.append(off[-1] + sub.n_i)
    assert (max(np.diff(off)) > 4693) == (m == 142)
    S.set_target(Z)
    net = a2ls.WarmStartNet(seed=3)
    theta = G.init_params(13).astype(np.float32).astype(np.float64)
    net.set_params(theta.astype(np.float32))
    Y = net.forward(S)
    params = G.unpack(theta)
    for i, (Aii, lump, n_I) in enumerate(inputs):
        Yo = G.forward(params, *G.graph_and_features(Aii, lump, n_I), bf16=True)["Y"]
        assert np.linalg.norm(Y[off[i]:off[i + 1]].astype(np.float64) - Yo) <= 1e-4 * np.linalg.norm(Yo)
    L, g = net.loss_grad(S), net.grads().astype(np.float64)
    Lo, go = G.sample_loss_grad(theta, [(*t, z) for t, z in zip(inputs, Z)], bf16=True)
    assert L == pytest.approx(Lo, rel=1e-4)
    o = 0
    for name, shape in G.param_shapes() if m != 142 else []:
        k = int(np.prod(shape))
        assert np.linalg.norm(g[o:o + k] - go[o:o + k]) <= 2e-3 * np.linalg.norm(go[o:o + k]) + 1e-9, name
        o += k
    net.close()
    S.close()
    P.close()


@pytest.mark.parametrize("lengths", [(3, 65, 64, 200), (16, 16, 16, 17), (1, 700, 33, 1000)])
def test_spmv_of_rows_far_apart_in_length(lengths):
    """Rows of the given lengths, one long one in 40: a thread's or a whole warp's where the rows are short on
    average, else four lanes'; the bound of the test above."""
    from paper_2201_02250_gb300 import a2ls
    n, r = 1003, np.random.default_rng(sum(lengths))
    A = sp.lil_matrix((n, n))
    for i in range(n):
        k = lengths[i % 4] if lengths[0] == 16 or i % 40 < 4 else lengths[0]
        cols = r.choice(n, min(k, n), replace=False)
        A[i, cols] = r.uniform(-1, 1, len(cols)) / n
    A = (A + sp.diags(np.full(n, 4.0))).tocsr()
    P, _keep = a2ls.from_scipy(A, (np.arange(n) * 4 // n).astype(np.int32), 0, 0, variant="ras")
    x = r.uniform(-1, 1, n)
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    P.spmv(torch.as_tensor(x, device="cuda"), y)
    bound = 2 * (max(lengths) + 1) * 2.0**-53 * (abs(A) @ abs(x))
    assert np.all(np.abs(y.cpu().numpy() - A @ x) <= bound)
