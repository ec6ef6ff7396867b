"""The FP64 path's reciprocal, square root and inverse cube root over the
whole range of exponents (their seeds handle exponents as integers and leave
subnormal, zero, negative and non-finite arguments to the plain functions):
within 1, 1 and 4 units in the last place of CUDA's IEEE results."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fp64_functions_over_all_exponents(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fp64_range_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-o", exe, os.path.join(HERE, "fp64_range_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    err = {k: float(v) for k, v in (line.split() for line in out.strip().splitlines())}
    assert err["rcp"] <= 1.0, err
    assert err["sqrt"] <= 1.0, err
    assert err["icbrt"] <= 4.0, err
    assert err["special"] == 0, err


def test_square_roots_are_correctly_rounded(tmp_path):
    """The FP64 path's square root is IEEE's, bit for bit, at the arguments
    whose roots are hardest to round too (tests/fp64_sqrt_check.cu)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fp64_sqrt_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-o", exe, os.path.join(HERE, "fp64_sqrt_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert out.strip() == "differ 0", out


def test_transposed_friction_takes_the_reciprocal_depth(tmp_path):
    """The depth part of the transposed friction holds 1 / h to an ulp
    (tests/fp64_vjp_check.cu): within two units in the last place."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fp64_vjp_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-o", exe, os.path.join(HERE, "fp64_vjp_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert int(out.split()[1]) <= 2, out


def test_the_time_step_is_the_ieee_quotient(tmp_path):
    """courant / rate, bit for bit (tests/fp64_dt_check.cu)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fp64_dt_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-o", exe, os.path.join(HERE, "fp64_dt_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert out.strip() == "differ 0", out
