"""The shared-A batch checks every vector that lies in host memory before it needs a device."""
import numpy as np
import pytest


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
