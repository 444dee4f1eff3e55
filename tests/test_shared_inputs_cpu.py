"""The shared-A batch checks every vector that lies in host memory before it needs a device, and gives
the device's room for the vectors back to a solve that has none
(tests/shared_vectors_check.cpp, linked with the library's own objects, answers the runtime's calls)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_vectors_move_to_the_host(tmp_path):
    from paper_1805_12344_gb300 import build
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    build.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    exe = tmp_path / "shared_vectors_check"
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", build.INCLUDE, "-o", str(exe),
                        os.path.join(HERE, "shared_vectors_check.cpp"), *objs, "-L", os.path.join(cuda, "lib64"), "-lcudart",
                        "-Wl,-rpath," + os.path.join(cuda, "lib64")], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr


@pytest.mark.parametrize("which", ["b", "c"])
def test_a_bad_host_vector_is_refused_without_a_device(which):
    from paper_1805_12344_gb300 import abip, build
    build.build()
    A = np.eye(2, 3)
    b, c = [np.ones(2) for _ in range(70)], [np.ones(3) for _ in range(70)]
    (b if which == "b" else c)[66][-1] = np.inf
    with pytest.raises(abip.AbipError) as e:
        abip.abip_solve_batch_shared(A, b, c)
    assert e.value.code == abip.ABIP_E_INVALID_ARG and "instance 66" in str(e.value)
