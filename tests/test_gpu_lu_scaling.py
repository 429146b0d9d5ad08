"""The double-float LU of badly scaled matrices (tests/cpp/lu_dfloat.cu), against extended precision."""
import os
import subprocess

import numpy as np
import pytest

from paper_2201_02250_gb300 import _build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
TB = 64   # columns of a step


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    path = str(tmp_path_factory.mktemp("lu") / "lu_dfloat")
    libdir = os.path.dirname(_build.LIB)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    os.path.join(HERE, "cpp", "lu_dfloat.cu"), "-L", libdir, "-lA2LS", "-Xlinker", "-rpath=" + libdir,
                    "-o", path], check=True)
    return path


def _lu(A):
    A = A.copy()
    for k in range(A.shape[0] - 1):
        A[k + 1:, k] /= A[k, k]
        A[k + 1:, k + 1:] -= np.outer(A[k + 1:, k], A[k, k + 1:])
    return np.tril(A, -1) + np.eye(A.shape[0], dtype=A.dtype), np.triu(A)


def _tri_inverse(T):
    """Inverse of a lower triangle."""
    X = np.eye(T.shape[0], dtype=T.dtype)
    for r in range(T.shape[0]):
        X[r] = (X[r] - T[r, :r] @ X[:r]) / T[r, r]
    return X


@pytest.mark.parametrize("tensor_cores", [0, 1])
@pytest.mark.parametrize("n,digits", [(97, 5), (330, 5), (330, 0)])
def test_panels_of_badly_scaled_matrices(exe, tmp_path, n, digits, tensor_cores):
    """Rows and columns scaled by random factors of 10^-digits to 10^digits: the first block column of L and block
    row of U have componentwise errors of rounding size, which scaling does not change.  With gamma = 64 u for the
    sums of up to 64 terms, u = 2^-46 a double-float operation: E = gamma |L||U| is the block's backward
    error, dU = |L^-1| E |U^-1| |U| (and dL likewise) what it does to U, and L21 = A21 U^-1 takes gamma for the product and the
    inverse and |dU| |U^-1| for U; four times that."""
    r = np.random.default_rng(n + digits)
    a, b = 10.0 ** r.uniform(-digits, digits, n), 10.0 ** r.uniform(-digits, digits, n)
    A = (np.where(np.eye(n) > 0, 0.6 * n, r.uniform(-1, 1, (n, n)))) * a[:, None] * b[None, :]
    hi = A.astype(np.float32).astype(np.float64)
    A = hi + (A - hi).astype(np.float32)      # values of 48 bits
    A.tofile(tmp_path / "a")
    subprocess.run([exe, str(n), str(tensor_cores), str(tmp_path / "a"), str(tmp_path / "f")], check=True, timeout=120)
    F = np.fromfile(tmp_path / "f").reshape(n, n)
    X = A.astype(np.longdouble)
    L, U = _lu(X[:TB, :TB])
    Li, Ui = _tri_inverse(L), _tri_inverse(U.T).T
    gamma = TB * 2.0**-46
    aL, aU, aLi, aUi = abs(L), abs(U), abs(Li), abs(Ui)
    E = gamma * (aL @ aU)
    # the factors of the block move by dU = |L^-1| E |U^-1| |U|, dL = |L| |L^-1| E |U^-1|
    dU, dL = aLi @ E @ aUi @ aU, aL @ aLi @ E @ aUi
    A21, A12 = X[TB:, :TB], X[:TB, TB:]
    boundL = abs(A21) @ (gamma * (aUi @ aU @ aUi) + aUi @ dU @ aUi)
    boundU = (gamma * (aLi @ aL @ aLi) + aLi @ dL @ aLi) @ abs(A12)
    errL, errU = abs(F[TB:, :TB] - A21 @ Ui) / boundL, abs(F[:TB, TB:] - Li @ A12) / boundU
    assert errL.max() <= 4 and errU.max() <= 4, (float(errL.max()), float(errU.max()))
