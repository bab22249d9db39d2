"""Function attributes are set once per device, not once per process (csrc/sp_device.h): the helper
runs on the CPU against a fake of the runtime's current device, and no source keeps such a flag of
its own."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1409_0297_gb300", "csrc")


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = tmp_path / "per_device"
    b = subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", cuda,
                        os.path.join(ROOT, "tests", "host", "per_device_main.cpp"), "-o", str(exe), "-lpthread"],
                       capture_output=True, text=True)
    assert b.returncode == 0, b.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


def test_no_flag_of_the_whole_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        with open(path) as f:
            assert not re.search(r"static bool\b", f.read()), path
