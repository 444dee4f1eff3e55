"""The FP64 group kernel at the sizes where its sums' parts change: one, two, four and eight parts,
fewer rows or columns than cells (nine to a part), and matrices that do not fit the shared memory of
16 CTAs (rows read from global memory).  First iterates against the oracle at the 1e-10 of the parity
tests; the same in a batch that gives every LP one CTA."""
import numpy as np
import pytest

from oracle import abip_oracle as O
from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
# (m, n): one part | two, fewer rows than cells | two | four | eight | 16 parts, two rows | 16, matrices not copied
SIZES = [(7, 20), (8, 70), (20, 40), (24, 100), (40, 120), (2, 1100), (225, 700)]


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


def _lps():
    return [W.planted_dense(m, n, seed=W.seed_for(W.DENSE_PLANTED, 1300 + m)) for m, n in SIZES]


def test_first_iterates_alone(abip):
    for lp in _lps():
        ref = O.run_iterations(lp.A, lp.b, lp.c, 8, O.Params(linsys=0))
        s = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=8)
        s.solve()
        assert _rel(s.stacked_state(), ref) <= TOL, lp.A.shape
        s.close()


def test_first_iterates_with_one_cta_each(abip):
    lps = _lps() + [W.planted_dense(12, 30, seed=W.seed_for(W.DENSE_PLANTED, 1400 + k)) for k in range(400)]
    infos, xs, ys, ss = abip.abip_solve_batch([l.A for l in lps], [l.b for l in lps], [l.c for l in lps],
                                              abip.default_params(max_admm_iters=8))
    for k, (m, n) in enumerate(SIZES):
        ref = O.run_iterations(lps[k].A, lps[k].b, lps[k].c, 8, O.Params(linsys=0))
        assert _rel(np.concatenate([ys[k], xs[k]]) * infos[k]["tau"], ref[:m + n]) <= TOL, (m, n)
