"""Device-side waits that run out end their kernel with an error status (tests/cpp/tc_solve_waits.cu)."""
import os
import subprocess

import pytest

from paper_2201_02250_gb300 import _build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_tensor_core_solve_gives_up_with_a_status(tmp_path):
    exe = str(tmp_path / "tc_solve_waits")
    libdir = os.path.dirname(_build.LIB)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    os.path.join(HERE, "cpp", "tc_solve_waits.cu"), "-L", libdir, "-lA2LS", "-Xlinker", "-rpath=" + libdir,
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
