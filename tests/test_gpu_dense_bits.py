"""A dense LP's result does not depend on what it is solved with: alone (Solver), in a batch of
itself, of a few, or of more LPs than the SMs take clusters of, the CTAs per LP range from 16 (or,
in FP64, the whole grid) to one, and the bits are the same.  Past an exact recomputation of the
mixed path's products (every 100 updates) and, for most of the LPs, a change of mu."""
import numpy as np
import pytest

from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UPDATES = 120
# (m, n): fewer rows than parts of the sums | 2 CTAs | 8 | 16 | odd | 16, matrices not copied to shared
# memory | the whole grid in FP64
SIZES = [(3, 7), (8, 70), (50, 120), (97, 97), (201, 611), (225, 700), (303, 905)]


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


def _lp(k):
    m, n = SIZES[k % len(SIZES)]
    return W.planted_dense(m, n, seed=W.seed_for(W.DENSE_PLANTED, 1100 + k))


def _batch(abip, lps, precision):
    prm = abip.default_params(max_admm_iters=UPDATES, precision=precision, eps=1e-12)
    infos, xs, ys, ss = abip.abip_solve_batch([l.A for l in lps], [l.b for l in lps], [l.c for l in lps], prm)
    return [(f["admm_iters"], f["outer_iters"], f["tau"], f["theta"], f["mu"], *x, *y, *s) for f, x, y, s in zip(infos, xs, ys, ss)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [2, 40, 700])
def test_bits_alone_and_in_a_batch(abip, precision, count):
    probe = [_lp(k) for k in range(len(SIZES))]
    alone = [_batch(abip, [lp], precision)[0] for lp in probe]
    assert any(a[1] > 0 for a in alone)
    fill = [W.planted_dense(20, 45, seed=W.seed_for(W.DENSE_PLANTED, 1200 + k)) for k in range(max(0, count - len(SIZES)))]
    if count == 2:
        for k, lp in enumerate(probe):
            assert _batch(abip, [probe[(k + 1) % len(probe)], lp], precision)[1] == alone[k], SIZES[k]
        return
    got = _batch(abip, probe + fill, precision)
    for k in range(len(SIZES)):
        assert got[k] == alone[k], SIZES[k]


@pytest.mark.parametrize("precision", [0, 1])
def test_bits_of_a_handle(abip, precision):
    for k, (m, n) in enumerate(SIZES):
        lp = _lp(k)
        want = _batch(abip, [lp], precision)[0]
        s = abip.Solver(lp.A, lp.b, lp.c, max_admm_iters=UPDATES, precision=precision, eps=1e-12)
        f, x, y, sv = s.solve()
        s.close()
        assert (f["admm_iters"], f["outer_iters"], f["tau"], f["theta"], f["mu"], *x, *y, *sv) == want, (m, n)
