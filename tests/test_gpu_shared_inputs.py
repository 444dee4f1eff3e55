"""The shared-A batch takes its inputs whole: every b and c is read and checked before the first of
the chunks of 64 instances is solved (a bad vector of a later chunk leaves nothing written, an
output may stand where a later instance's input stood), and a row count that does not fit a grid's
y extent (n above 32 * 65535) is solved like any other."""
import ctypes as C

import numpy as np
import pytest

from oracle import abip_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

M, N, COUNT = 4, 9, 70   # two chunks


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


def _lps():
    rng = np.random.default_rng(31)
    A = rng.standard_normal((M, N))
    b = rng.uniform(0.5, 2.0, (COUNT, N)) @ A.T
    c = rng.standard_normal((COUNT, M)) @ A + rng.uniform(0.5, 2.0, (COUNT, N))
    return A, b, c


def _call(abip, A, b, c, x, prm):
    """abip_solve_batch_shared on rows of b, c and x (numpy arrays or CUDA tensors); the return code."""
    def ptrs(rows):
        return (C.c_void_p * len(rows))(*[abip._ptr(r)[0] for r in rows])
    Mx, keep = abip._matrix(A)
    infos = (abip.abip_info * len(b))()
    for f in infos:
        f.status = -7
    rc = abip.lib().abip_solve_batch_shared(len(b), C.byref(Mx), ptrs(b), ptrs(c), C.byref(prm), ptrs(x), None, None, infos, None)
    return rc, [f.status for f in infos]


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("which", ["b", "c"])
def test_a_bad_vector_of_a_later_chunk_leaves_nothing_written(abip, device, which):
    A, b, c = _lps()
    (b if which == "b" else c)[66, -1] = np.nan
    x = np.full((COUNT, N), 123.0)
    if device:
        A, b, c, x = (torch.from_numpy(t).cuda() for t in (A, b, c, x))
    rc, status = _call(abip, A, list(b), list(c), list(x), abip.default_params(max_admm_iters=3))
    assert rc == abip.ABIP_E_INVALID_ARG
    assert "instance 66" in abip.lib().abip_last_error(None).decode()
    assert all(s == -7 for s in status)
    assert bool((x == 123.0).all())


@pytest.mark.parametrize("device", [False, True])
def test_an_output_may_stand_where_a_later_input_stood(abip, device):
    A, b, c = _lps()
    prm = abip.default_params(max_admm_iters=3)
    want = np.stack(abip.abip_solve_batch_shared(A, list(b), list(c), prm)[1])
    x = np.zeros((COUNT, N))
    if device:
        A, b, c, x = (torch.from_numpy(t).cuda() for t in (A, b, c, x))
    rows = list(x)
    rows[:6] = list(c)[64:]   # the first six x go where the last six c are
    rc, _ = _call(abip, A, list(b), list(c), rows, prm)
    assert rc == abip.ABIP_OK
    got = np.stack([r.cpu().numpy() if device else r for r in rows])
    assert np.array_equal(got, want)


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
