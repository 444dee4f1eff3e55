"""FP64 sparse path: the lanes per row follow the grid's threads; the iterates do not.

`grid_ctas = 1` leaves 768 lanes, so rows keep the lanes that 16 entries each give them; the
default grid gives small LPs up to 32 per row.  Both solve each projection to cg_tol, so after
`updates` updates they differ by at most about updates * 2 * cg_tol * |q| (|q| < 1e3 here)."""
import numpy as np
import pytest

from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


def _lp(kind, m):
    if kind == "sparse":
        lp = W.planted_sparse(m, seed=7)
        return lp.A, lp.b, lp.c
    lp = W.planted_dense(m, 3 * m + 1, seed=7)   # every row longer than 32 lanes of 4 entries from m = 43 on
    return W.dense_to_csr(lp.A), lp.b, lp.c


@pytest.mark.parametrize("kind,m", [("sparse", 9), ("sparse", 33), ("sparse", 767), ("sparse", 2500), ("rows", 5), ("rows", 47)])
def test_iterates_do_not_follow_the_lanes(abip, kind, m):
    A, b, c = _lp(kind, m)
    out = []
    for ctas in (1, 0):
        s = abip.Solver(A, b, c, grid_ctas=ctas, cg_tol=1e-13, max_admm_iters=20)
        info, x, y, sl = s.solve()
        s.close()
        out.append((info["status"], info["admm_iters"], np.concatenate([x, y, sl])))
    assert out[0][:2] == out[1][:2]
    assert np.linalg.norm(out[0][2] - out[1][2]) <= 20 * 2 * 1e-13 * 1e3 * max(1.0, np.linalg.norm(out[0][2]))
