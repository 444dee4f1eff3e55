"""The sparse direct projection by its two routes: the group kernel with the inverse of the dense
factor (at most 1600 rows, grid_ctas = 0) and the factor's sweeps on the persistent grid, which
grid_ctas > 0 asks for at any size.  First iterates against the oracle at the 1e-10 of the parity
tests, a second solve and a resumed one on the same handle, ends and infeasible statuses, and the
wait limit as an error."""
import numpy as np
import pytest

from oracle import abip_oracle as O
from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
ROUTES = [0, 6]   # grid_ctas: the group kernel | the sweeps on six CTAs


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


def _solver(abip, A, b, c, ctas, **kw):
    return abip.Solver(A, b, c, linsys=abip.ABIP_LINSYS_SPARSE_LDL, grid_ctas=ctas, **kw)


@pytest.mark.parametrize("ctas", ROUTES)
def test_the_route_follows_grid_ctas(abip, ctas):
    """The group kernel is one launch; beside the sweeps' kernel there are others (start, scaled outputs)."""
    lp = W.grid_flow(6)
    s = _solver(abip, lp.A, lp.b, lp.c, ctas, max_admm_iters=5)
    info, *_ = s.solve()
    s.close()
    assert (info["launches"] == 1) == (ctas == 0)


@pytest.mark.parametrize("ctas", ROUTES)
def test_second_solve_and_resumed_solve(abip, ctas):
    lp = W.planted_sparse(300, seed=W.seed_for(W.SPARSE_PLANTED, 20))
    ref = O.run_iterations(lp.A.to_scipy(), lp.b, lp.c, 20, O.Params(linsys=0))
    s = _solver(abip, lp.A, lp.b, lp.c, ctas, max_admm_iters=20)
    s.solve()
    first = s.stacked_state()
    assert _rel(first, ref) <= TOL
    s.solve()
    assert _rel(s.stacked_state(), first) <= 1e-13
    s.close()
    half = _solver(abip, lp.A, lp.b, lp.c, ctas, max_admm_iters=10)
    half.solve()
    half.set_state(half.state())
    half.solve()
    assert _rel(half.stacked_state(), ref) <= TOL
    half.close()


@pytest.mark.parametrize("ctas", ROUTES)
def test_grid_flow_end_to_end(abip, ctas, oracle_memo):
    lp = W.grid_flow(6)
    ref = oracle_memo(("grid_flow", 6), lambda: O.solve(lp.A.to_scipy(), lp.b, lp.c, O.Params(linsys=0)))
    s = _solver(abip, lp.A, lp.b, lp.c, ctas)
    info, x, _, _ = s.solve()
    s.close()
    assert info["status"] == ref.status == O.OPTIMAL
    assert max(info["pres"], info["dres"], info["dgap"]) <= 1e-6
    assert abs(info["obj"] - ref.obj) <= 1e-5 * max(1.0, abs(ref.obj))
    assert np.linalg.norm(lp.A.to_dense() @ x - lp.b) <= 1.01e-6 * (1 + np.linalg.norm(lp.b))


@pytest.mark.parametrize("ctas", ROUTES)
@pytest.mark.parametrize("make", [W.infeasible_twin, W.dual_infeasible])
def test_infeasible_status(abip, ctas, make):
    lp = make()
    s = _solver(abip, W.dense_to_csr(lp.A), lp.b, lp.c, ctas)
    info, *_ = s.solve()
    s.close()
    assert info["status"] == O.solve(lp.A, lp.b, lp.c).status


@pytest.mark.parametrize("ctas", ROUTES)
def test_wait_limit_is_an_error(abip, ctas):
    lp = W.grid_flow(6)
    with pytest.raises(abip.AbipError) as e:
        _solver(abip, lp.A, lp.b, lp.c, ctas, barrier_limit_ns=1).solve()
    assert e.value.code == abip.ABIP_E_TIMEOUT
    s = _solver(abip, lp.A, lp.b, lp.c, ctas, max_admm_iters=5)
    assert s.solve()[0]["admm_iters"] == 5
    s.close()
