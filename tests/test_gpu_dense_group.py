"""The FP64 dense solve by a group of CTAs: every cluster size of the dispatch, the whole-grid
form, ranks without rows or columns (m or n below the CTAs), odd sizes (padded rows), copies in
shared memory or not, a resumed state and the other warm start.  First iterates against the
oracle at the 1e-10 of the parity tests; a run resumed from its own state continues it within
the same bound."""
import numpy as np
import pytest

from oracle import abip_oracle as O
from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# one CTA | 2 | 8 | 16, one row | 16 | 16, no matrix copies | grid, fewer rows than CTAs | grid, odd
@pytest.mark.parametrize("m,n", [(2, 3), (9, 31), (50, 121), (1, 3001), (97, 97), (201, 611), (61, 4400), (303, 905)])
@pytest.mark.parametrize("warmstart", [0, 1])
def test_first_iterates(abip, m, n, warmstart):
    lp = W.planted_dense(m, n, seed=W.seed_for(W.DENSE_PLANTED, 900 + m))
    ref = O.run_iterations(lp.A, lp.b, lp.c, 8, O.Params(linsys=0, warmstart=warmstart))
    s = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=8, warmstart=warmstart)
    s.solve()
    assert _rel(s.stacked_state(), ref) <= TOL
    s.close()


@pytest.mark.parametrize("m,n", [(33, 90), (303, 905)])
def test_resumed_run_continues(abip, m, n):
    lp = W.planted_dense(m, n, seed=W.seed_for(W.DENSE_PLANTED, 950 + m))
    whole = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=30)
    whole.solve()
    part = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=15)
    part.solve()
    part.set_state(part.state())
    part.solve()
    assert _rel(part.stacked_state(), whole.stacked_state()) <= TOL
    whole.close()
    part.close()


@pytest.mark.parametrize("count", [3, 40, 80])
def test_batch_first_iterates(abip, count):
    lps = [W.planted_dense(8 + (5 * k) % 60, 70 + k, seed=W.seed_for(W.DENSE_PLANTED, 1000 + k)) for k in range(count)]
    infos, xs, ys, ss = abip.abip_solve_batch([l.A for l in lps], [l.b for l in lps], [l.c for l in lps],
                                              abip.default_params(max_admm_iters=8))
    for k in range(0, count, 7):
        ref = O.run_iterations(lps[k].A, lps[k].b, lps[k].c, 8, O.Params(linsys=0))
        m, n = lps[k].A.shape
        assert _rel(np.concatenate([ys[k], xs[k]]) * infos[k]["tau"], ref[:m + n]) <= TOL, k


def test_grid_barrier_limit_is_an_error(abip):
    """A grid barrier that cannot be met in 1 ns ends the call with the timeout code; the handle of
    another solve works afterwards."""
    lp = W.planted_dense(303, 905, seed=W.seed_for(W.DENSE_PLANTED, 960))
    s = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=200, barrier_limit_ns=1)
    with pytest.raises(abip.AbipError) as e:
        s.solve()
    assert e.value.code == abip.ABIP_E_TIMEOUT
    s.close()
    ok = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=5)
    assert ok.solve()[0]["admm_iters"] == 5
    ok.close()
