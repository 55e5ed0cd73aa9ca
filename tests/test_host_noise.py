"""The white noise of the initial conditions (csrc/ic_noise.cuh), which takes its
logarithm, root and cosine from tables and short series, on the host against long
double (host/noise_check.cu)."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

# Largest errors in units of 2^-53 (half a last place at 1).  Logarithm, relative:
# table value, inner sum and outer sum rounded once each.  Root: the last step.
# Cosine, absolute: table value and sum, and their small terms.  Noise: g up to 8.6
# times the cosine's error, half the logarithm's, the root's and the product's.
BOUNDS = {"log": 3.0, "root": 1.5, "cos": 2.0, "noise": 8.6 * (2.0 + 1.5 + 1.5 + 1.0), "double": 0.0}


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("noise") / "noise_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "host", "noise_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {name: float(v) for name, v in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("name", sorted(BOUNDS))
def test_noise_functions(errors, name):
    assert errors[name] <= BOUNDS[name]
