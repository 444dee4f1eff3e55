"""The backward's elimination of columns before the LU: none eliminated (entries of A above every
s_j / x_j), all (entries of A and c below them), some, with core orders at and around the 32-wide
panels.  Against the oracle's gradient at the same point with the tolerance of the other
backward tests (1e-5 relative per block)."""
import numpy as np
import pytest

from oracle import abip_oracle as O
from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-5


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


@pytest.mark.parametrize("m,n,scale,cap", [(1, 2, 1.0, 30), (9, 21, 1e3, 20), (9, 21, 1e-3, 20), (15, 40, 1.0, 40),
                                           (31, 62, 1.0, 60), (33, 70, 1.0, 60)])
def test_gradient_with_some_none_and_all_columns_eliminated(abip, m, n, scale, cap):
    lp = W.planted_dense(m, n, seed=W.seed_for(W.DENSE_PLANTED, 1200 + m))
    A, b, c = lp.A * scale, lp.b * scale, lp.c * (scale if scale < 1 else 1.0)
    s = abip.Solver(A, b, c, max_admm_iters=cap)
    info, x, _, _ = s.solve()
    g = np.cos(np.arange(n))
    out = s.backward(g)
    st = s.state()
    start = dict(y=st[:m], x=st[m:m + n], tau=st[m + n], theta=st[m + n + 1], s=st[m + n + 2:m + 2 * n + 2],
                 kappa=st[m + 2 * n + 2])
    ref = O.central_point_grad(A, b, c, st[-1], lambda xs: g, start=start)
    for k, key in (("c", "dc"), ("b", "db"), ("A", "dA")):
        err = np.abs(out[k] - ref[key]).max() / np.abs(ref[key]).max()
        assert err <= GRAD_TOL, (k, err)
    s.close()
