"""The FP64 group kernel's barrier step, compiled for the host (tests/barrier_refined_check.cpp): both
roots within the derived 2.5 and 3.5 roundings of the closed form, over the range and at its ends."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_refined_barrier_step_is_within_its_roundings(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "barrier_refined_check"
    r = subprocess.run([gxx, "-std=c++17", "-O2", "-Wall", "-o", str(exe), os.path.join(HERE, "barrier_refined_check.cpp")],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout[:2000] + r.stderr
