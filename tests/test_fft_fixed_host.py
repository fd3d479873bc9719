"""The fixed-point line FFTs of the FP64 path (csrc/fixed.cuh), compiled for the host through
their __host__ paths: every supported length, both directions, on integers whose absolute sum
fills the 2^61 bound, against the exact integer DFT; the compile-time constants against the
host's cosine; the 64-bit product at its range's ends."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_line_ffts_match_the_exact_dft(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "fft_fixed"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O2",
                    "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1611_06797_gb300", "csrc"), "-x", "cu",
                    os.path.join(ROOT, "tests", "native", "fft_fixed.cu"), "-o", str(exe)],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    rows = [line.split() for line in out.strip().splitlines()]
    ffts = [r for r in rows if r[0].isdigit()]
    assert {int(r[0]) for r in ffts} == {8, 10, 12, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40}
    assert len(ffts) == 26
    for n, d, units in ffts:
        # A stage rounds each value at most four times (three shears or products of at most half
        # a unit, one halving below a unit) and later stages pass an error on with the weights of
        # a DFT over the stages left: at most 2.5 sqrt(n) units, and 0.2 units from the constants
        # (2^-61 of a value below 2^61)
        assert float(units) <= 2.5 * int(n) ** 0.5 + 0.2, (n, d, units)
    const = float(next(r for r in rows if r[0] == "const")[2])
    assert const < 2.0 ** -59, const           # long double cosine: 2^-64 on x86, 2^-53 where it is a double
    mean, worst, back = map(float, next(r for r in rows if r[0] == "mul")[1:])
    # rounding to nearest (half a unit) and the dropped product of the low halves (half a unit)
    assert worst < 1.01 and abs(mean) < 0.01 and back == 0


def test_packed_line_ffts_match_the_dft(tmp_path):
    """The FP32 transforms of two lines at once (csrc/pair.cuh), compiled for the host."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "fft_pair"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O2",
                    "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1611_06797_gb300", "csrc"), "-x", "cu",
                    os.path.join(ROOT, "tests", "native", "fft_pair.cu"), "-o", str(exe)],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    rows = [line.split() for line in out.strip().splitlines()]
    assert {int(r[0]) for r in rows} == {8, 10, 12, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40} and len(rows) == 26
    for n, d, err in rows:
        # at most log2(n) butterfly stages of at most 4 roundings (2^-24 each) on a value
        assert float(err) <= 4 * 2.0 ** -24 * int(n).bit_length(), (n, d, err)
