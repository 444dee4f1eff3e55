"""Inputs of the shared-A batch: a column count whose blocks of 32 do not fit a grid's y extent (n
above 32 * 65535) is solved like any other."""
import numpy as np
import pytest

from oracle import abip_oracle as O

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


def test_more_columns_than_a_grids_y_extent_holds(abip):
    """First iterates against the oracle at the 1e-10 of the parity tests."""
    m, n, k = 2, 32 * 65535 + 33, 3
    rng = np.random.default_rng(32)
    A = rng.standard_normal((m, n))
    b = A @ rng.uniform(0.5, 2.0, n)
    c = A.T @ rng.standard_normal(m) + rng.uniform(0.5, 2.0, n)
    infos, xs, ys, ss = abip.abip_solve_batch_shared(A, [b], [c], abip.default_params(max_admm_iters=k))
    f = infos[0]
    got = np.concatenate([ys[0] * f["tau"], xs[0] * f["tau"], [f["tau"], f["theta"]], ss[0] * f["tau"], [f["kappa"]]])
    ref = O.run_iterations(A, b, c, k, O.Params(linsys=0))
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
