"""The fixed-point arithmetic of the FP64 FFT passes (csrc/fft_fixed.cuh),
compiled for the CPU: every radix against extended precision.

Bound: a chain of two small DFTs, a twiddle and two factors rounds four times,
each by at most 2^-56 of the 2-norm of the vector (58-bit components aligned
to the largest, which is at most the 2-norm; products to one unit of 2^-57 of
the vector's scale), and the final alignment rounds down by half a unit on
average: below 2^-53 of the result's 2-norm in all, which is what one
rounding to a double costs."""
import math
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0809_3739_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("fx") / "fixed_point_host")
    subprocess.run([NVCC, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-o", exe, os.path.join(HERE, "fixed_point_host.cu")], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()


def test_every_radix_within_half_an_ulp(lines):
    seen = 0
    for line in lines:
        w = line.split()
        if w[0].isdigit():
            assert float(w[2]) < 2.0 ** -53, line
            seen += 1
    assert seen == 7 * 6


@pytest.mark.parametrize("name,x,y", [
    ("zero", 0.0, 0.0), ("subnormal", 0.0, 0.0), ("large", 1.5e300, 3e300),
    ("small", 1.5e-300, -3e-300), ("one", 1.5, -6.0)])
def test_special_values(lines, name, x, y):
    w = next(line.split() for line in lines if line.startswith(name))
    for got, want in ((float(w[1]), x), (float(w[2]), y)):
        assert math.isclose(got, want, rel_tol=2.0 ** -52, abs_tol=0.0)


@pytest.mark.parametrize("name", ["nan", "inf"])
def test_non_finite_values_spread(lines, name):
    w = next(line.split() for line in lines if line.startswith(name))
    assert math.isnan(float(w[1])) and math.isnan(float(w[2]))
