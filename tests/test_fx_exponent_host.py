"""Exponents of the FP64 path's fixed-point co-densities (csrc/fixed.cuh): a state's exponent is at or above
that of each of its planes, so that the shift between the two is never negative: the exponent may not
fall as the norm grows."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_exponents_rise_with_the_norm(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "fx_exponent"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O2",
                    "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1611_06797_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "fx_exponent.cu"), "-o", str(exe)],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    falls, bound, zero, nan, inf = map(int, out)
    assert falls == 0 and bound == 0
    assert zero == -480 and nan == 1 and inf == 1
