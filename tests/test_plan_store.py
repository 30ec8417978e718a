"""The device copies of a mesh's patch plans on the CPU, against a fake of the
CUDA runtime (tests/plan_store_check.cpp): failed uploads, sharing, idle
copies and the order in which they are freed."""
import os
import shutil
import subprocess

import pytest

from paper_2105_13484_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_plan_store(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    out = str(tmp_path / "plan_store_check")
    r = subprocess.run([gxx, "-O1", "-std=c++17", "-pthread", "-I", inc, "-o", out,
                        os.path.join(HERE, "plan_store_check.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([out], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
