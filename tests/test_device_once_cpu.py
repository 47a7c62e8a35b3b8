"""Kernel attributes are set once per device (csrc/device_once.cuh), not once per process: with a process-wide flag the second
device's first tensor-core product was refused for its shared memory."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_17898_gb300", "csrc")


def test_each_device_by_itself(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "device_once_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I", CSRC, os.path.join(ROOT, "tests", "native", "device_once_check.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


def test_no_process_wide_flag_in_the_launchers():
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static bool \w+ = false;\s*if \(!\w+\) \{\s*(const )?cudaError_t \w+ = cudaFuncSetAttribute", text), name
