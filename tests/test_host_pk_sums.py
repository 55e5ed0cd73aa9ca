"""The shell sums of the power spectrum (csrc/pk_sums.cuh) on the host against long
double (host/pk_sums_check.cu)."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

# In units of 2^-53 of the sum.  Its double: two conversions and a sum, 1/2 each.  Each
# square is rounded at 2^-61 (2^-59 in `small`) of the largest one, which a sum of n
# modes holds at least once: 2 n 2^-61 2^53 < 16 for 2048 modes of very different sizes,
# less than 1 for up to 512, and next to nothing where all are alike.
BOUNDS = {"one": 2.0, "wide": 18.0, "holes": 18.0, "small": 18.0}


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("pk_sums") / "pk_sums_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "host", "pk_sums_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {name: float(v) for name, v in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("name", sorted(BOUNDS))
def test_sums_of_squares(errors, name):
    # (squares rounded to float32 would be 2^28 off one by one, and 2^23 in such sums)
    assert errors[name] <= BOUNDS[name]
