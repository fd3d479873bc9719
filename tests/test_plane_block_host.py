"""The FP64 plane kernel's block (csrc/plane_block.h) is made of whole warps for every grid and every
number of planes that a caller or the autotuner may ask for: its sum over the block reads every lane
of every warp."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_blocks_are_whole_warps(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = tmp_path / "plane_block"
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1611_06797_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "plane_block.cpp"), "-o", str(exe)], check=True)
    rows = [tuple(map(int, line.split())) for line in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 13 * 64
    for n, ask, ib, threads in rows:
        assert threads % 32 == 0 and 64 <= threads <= 256, (n, ask, ib, threads)
        assert 1 <= ib <= ask and threads >= ib * n, (n, ask, ib, threads)
        assert ib == ask or (ib + 1) * n > 256, (n, ask, ib, threads)
