"""Shared-memory limits of kernels do not follow the call, on the CPU: tests/smem_limit_check.cpp is
linked with the library's own objects and answers the runtime's calls itself; and no source sets such
a limit to a value of the call."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_the_inverses_limit_is_the_same_for_every_call(tmp_path):
    from paper_1805_12344_gb300 import build
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    build.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    exe = tmp_path / "smem_limit_check"
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", build.INCLUDE, "-o", str(exe),
                        os.path.join(HERE, "smem_limit_check.cpp"), *objs, "-L", os.path.join(cuda, "lib64"), "-lcudart",
                        "-Wl,-rpath," + os.path.join(cuda, "lib64")], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr


def test_every_limit_is_a_constant():
    from paper_1805_12344_gb300 import build
    found = 0
    for name in sorted(os.listdir(build.CSRC)):
        if not name.endswith(".cu"):
            continue
        with open(os.path.join(build.CSRC, name)) as f:
            text = f.read()
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*\(int\)\s*(\S+?)\)", text):
            found += 1
            assert re.fullmatch(r"(tc::)?k[A-Z]\w*", m.group(1)), (name, m.group(0))
    assert found >= 10
