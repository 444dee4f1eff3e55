"""The way down from clusters that a device does not hold, on the CPU: tests/cluster_plan_check.cpp is
linked with the library's own objects and answers the runtime's calls itself."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_plans_follow_the_clusters_that_fit(tmp_path):
    from paper_1805_12344_gb300 import build
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    build.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    exe = tmp_path / "cluster_plan_check"
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", build.INCLUDE, "-o", str(exe),
                        os.path.join(HERE, "cluster_plan_check.cpp"), *objs, "-L", os.path.join(cuda, "lib64"), "-lcudart",
                        "-Wl,-rpath," + os.path.join(cuda, "lib64")], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
