"""The double-float Schur iteration of the mixed set-ups, on the host (tests/cpp/small_eig_dfloat.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    tmp = tmp_path_factory.mktemp("se")
    path = str(tmp / "small_eig_dfloat")
    (tmp / "cuda_runtime.h").write_text("")   # the source brings what it needs of it
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", str(tmp),
                    os.path.join(HERE, "cpp", "small_eig_dfloat.cpp"), "-o", path], check=True)
    return path


def _matrix(kind, m, rng):
    H = rng.standard_normal((m, m))
    if kind == "rotations":       # complex pairs only, of moduli from 1 to 1e-8
        H = np.zeros((m, m))
        for j in range(0, m - 1, 2):
            r, a = 10.0 ** rng.uniform(-8, 0), rng.uniform(0.1, 3)
            H[j:j + 2, j:j + 2] = r * np.array([[np.cos(a), -np.sin(a)], [np.sin(a), np.cos(a)]])
        X = np.linalg.qr(rng.standard_normal((m, m)))[0]
        H = X @ H @ X.T
    elif kind == "tiny_subdiagonal":   # Hessenberg, with subdiagonal entries whose squares FP32 cannot hold
        H = np.triu(H, -1)
        i = np.arange(m - 1)
        H[i + 1, i] *= np.where(rng.uniform(size=m - 1) < 0.5, 10.0 ** rng.uniform(-24, -10, m - 1), 1.0)
    elif kind == "small":
        H *= 1e-13
    elif kind == "large":
        H *= 1e12
    elif kind == "graded":
        H = H * 10.0 ** -np.linspace(0, 12, m)[:, None]
    return H


@pytest.mark.parametrize("kind", ["random", "rotations", "tiny_subdiagonal", "small", "large", "graded"])
def test_schur_form_is_orthogonal_and_backward_stable(exe, kind):
    """An entry of Q or H is touched by up to about 3 m^2 reflections (three sweeps an eigenvalue), each of which
    leaves a relative error of at most 8 u, u = 2^-47; added up like a random walk and with a factor of four,
    32 sqrt(3) m u for Q^T Q - I, and m^(1/2) times the largest entry of H (its columns' norms) as often for H."""
    rng = np.random.Generator(np.random.PCG64(len(kind)))
    for m in (2, 3, 5, 17, 32, 47, 72, 96):
        H = _matrix(kind, m, rng)
        r = subprocess.run([exe], input=f"{m}\n" + "\n".join(" ".join(f"{v:.17g}" for v in row) for row in H),
                           capture_output=True, text=True, check=True)
        out = np.array(r.stdout.split(), dtype=np.float64)
        rc, orth, back, hn = out[:4]
        ev = out[4::2] + 1j * out[5::2]
        tol = 32 * np.sqrt(3) * m * 2.0**-47
        assert rc == 0
        assert orth <= tol and back <= tol * np.sqrt(m) * hn, (m, orth / tol, back / (tol * np.sqrt(m) * hn))
        # trace: the sum of the eigenvalues, to the backward error of m diagonal entries
        assert abs(ev.sum() - np.trace(H)) <= m * tol * np.sqrt(m) * hn
