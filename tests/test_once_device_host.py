"""Per-device set-up (csrc/once_device.h): the exact-slice product's shared-memory limit belongs to
one device, so it is set once for each and not once for the process, and a failure is not kept."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1611_06797_gb300", "csrc")


def test_once_for_each_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = tmp_path / "once"
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, os.path.join(ROOT, "tests", "native", "once_device.cpp"),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert out.splitlines() == ["devices 1 1", "retry 2 2 0 0", "threads 1 1 1 1 early 0", "beyond 3"]


def test_no_process_wide_flag_guards_device_state():
    """No set-up of a device hangs on a flag of the process."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert "once_flag" not in text and "call_once" not in text, name
