"""The sparse direct projection with the inverse of the dense factor (LPs of at most 1600 rows,
solved by a group of CTAs over the CSR entries) and, above that, with the sparse factor's sweeps:
one CTA, clusters with and without copies in shared memory, the whole grid, entries given twice,
a resumed state.  First iterates against the oracle at the 1e-10 of the parity tests."""
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


def _first(abip, A, b, c, k):
    s = abip.Solver(A, b, c, linsys=abip.ABIP_LINSYS_SPARSE_LDL, max_admm_iters=k)
    s.solve()
    got = s.stacked_state()
    s.close()
    return got


@pytest.mark.parametrize("side", [2, 5, 16, 24, 33, 41])   # 41: m = 1680, the sweeps
def test_grid_flow_first_iterates(abip, side):
    lp = W.grid_flow(side)
    ref = O.run_iterations(lp.A.to_scipy(), lp.b, lp.c, 8, O.Params(linsys=0))
    assert _rel(_first(abip, lp.A, lp.b, lp.c, 8), ref) <= TOL


def test_duplicate_entries_add_up(abip):
    """Each entry of a random sparse A split into two stored entries, in no column order."""
    lp = W.planted_sparse(40, seed=W.seed_for(W.SPARSE_PLANTED, 41))
    A = lp.A
    rng = np.random.default_rng(3)
    ci, va, rp = [], [], [0]
    for i in range(A.m):
        k = slice(A.row_ptr[i], A.row_ptr[i + 1])
        part = rng.uniform(0.1, 0.9, A.row_ptr[i + 1] - A.row_ptr[i])
        col = np.concatenate([A.col_idx[k], A.col_idx[k]])
        val = np.concatenate([A.val[k] * part, A.val[k] * (1 - part)])
        order = rng.permutation(col.size)
        ci.append(col[order]); va.append(val[order]); rp.append(rp[-1] + col.size)
    B = W.CSR(m=A.m, n=A.n, row_ptr=np.asarray(rp), col_idx=np.concatenate(ci).astype(np.int32),
              val=np.concatenate(va).astype(np.float64))
    ref = O.run_iterations(B.to_scipy(), lp.b, lp.c, 8, O.Params(linsys=0))
    assert _rel(_first(abip, B, lp.b, lp.c, 8), ref) <= TOL


def test_resumed_run_continues(abip):
    lp = W.grid_flow(9)
    whole = _first(abip, lp.A, lp.b, lp.c, 30)
    s = abip.Solver(lp.A, lp.b, lp.c, linsys=abip.ABIP_LINSYS_SPARSE_LDL, max_admm_iters=15)
    s.solve()
    s.set_state(s.state())
    info, x, y, sv = s.solve()
    assert _rel(s.stacked_state(), whole) <= TOL
    st = s.state()
    assert np.array_equal(x * info["tau"], x * st[lp.m + lp.n]) and info["mu"] == st[-1]
    s.close()
