"""The integer scalars of the dense kernels (csrc/fx_scalar.cuh), compiled for
the CPU, against extended precision.

Bounds: reciprocals, inverse square roots and the reflector's scalars carry
2^-60 or better before they are rounded to a double, so their relative error is
below 1.02 * 2^-53; a sum of 32 addends, each rounded to half a unit of 2^-57 of
the largest, is off by 32 of those (and the rounding of the result)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0809_3739_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("fx") / "dense_scalars_host")
    subprocess.run([NVCC, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-o", exe, os.path.join(HERE, "dense_scalars_host.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {k: float(v) for k, v in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("name,bound", [("recip", 1.02), ("rsqrt", 1.02), ("alpha", 1.02),
                                        ("v0", 1.02), ("beta", 1.02), ("sum", 1.0)])
def test_scalar(errors, name, bound):
    assert errors[name] <= bound, errors
