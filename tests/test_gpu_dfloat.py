"""Double-float arithmetic of the device against exact values (tests/cpp/dfloat_device.cu)."""
import os
import subprocess

import pytest

from paper_2201_02250_gb300 import _build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_reciprocals_and_digits(tmp_path):
    """rsqrt: the residual 1 - a y^2 takes two products and a subtraction of 2^-47 each and is halved, the last sum
    rounds to 2^-48; recip: one product less, not halved: both at most four times 2^-47.  The digits round the two
    halves of a value to integers, at most 2^-56 of the scale together."""
    exe = str(tmp_path / "dfloat_device")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    os.path.join(HERE, "cpp", "dfloat_device.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    rsqrt, recip, digits, bad = (float(v) for v in r.stdout.split())
    assert rsqrt <= 4 and recip <= 4 and digits <= 1 and bad == 0, r.stdout
