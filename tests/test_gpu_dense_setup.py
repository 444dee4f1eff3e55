"""The dense setup split over the SMs (Gram tiles, cluster Cholesky, column-tiled inverse) at the
edges of its 32-wide blocks and of its dispatch: one instance (8-CTA clusters, 4-column inverse
tiles), a few (8-column tiles) and more than twice the SMs (32-column tiles).

FP64 iterates agree with the oracle to the 1e-10 of the parity tests.  A mixed update is formed
from FP32 products of changes of order 1, each off by at most n 2^-24 relative: 4 updates at
n <= 200 stay within 1e-4 of the FP64 iterate."""
import numpy as np
import pytest

from oracle import abip_oracle as O
from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UPDATES = 4


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


@pytest.mark.parametrize("m", [1, 31, 32, 33, 64, 65, 97])
def test_single_instance_first_iterates(abip, m):
    lp = W.planted_dense(m, 2 * m + 3, seed=W.seed_for(W.DENSE_PLANTED, 700 + m))
    ref = O.run_iterations(lp.A, lp.b, lp.c, UPDATES, O.Params(linsys=0))
    for precision, tol in ((abip.ABIP_PREC_F64, 1e-10), (abip.ABIP_PREC_MIXED, 1e-4)):
        s = abip.Solver(lp.A, lp.b, lp.c, precision=precision, max_admm_iters=UPDATES)
        s.solve()
        assert _rel(s.stacked_state(), ref) <= tol, (m, precision)
        s.close()


@pytest.mark.parametrize("count", [90, 320])
def test_batch_first_iterates(abip, count):
    sizes = [(1 + (7 * k) % 67, k) for k in range(count)]
    lps = [W.planted_dense(m, 2 * m + k % 5, seed=W.seed_for(W.DENSE_PLANTED, 800 + k)) for m, k in sizes]
    args = ([l.A for l in lps], [l.b for l in lps], [l.c for l in lps])
    for precision, tol in ((abip.ABIP_PREC_F64, 1e-10), (abip.ABIP_PREC_MIXED, 1e-4)):
        infos, xs, ys, ss = abip.abip_solve_batch(*args, abip.default_params(precision=precision, max_admm_iters=UPDATES))
        for k in range(0, count, 13):
            ref = O.run_iterations(lps[k].A, lps[k].b, lps[k].c, UPDATES, O.Params(linsys=0))
            m, n = lps[k].A.shape
            got = np.concatenate([ys[k], xs[k]]) * infos[k]["tau"]
            assert _rel(got, ref[:m + n]) <= tol, (k, precision)


@pytest.mark.parametrize("precision", [0, 1])
def test_device_inputs_equal_host_inputs(abip, precision):
    """A, b, c on the device (FP32 or FP64 A, odd sizes) give the bits of the same values from the host."""
    lp = W.planted_dense_f32(33, 71, seed=11)
    A, b, c = (torch.from_numpy(v).cuda() for v in (lp.A, lp.b, lp.c))
    states = []
    for args in ((lp.A, lp.b, lp.c), (A, b, c), (A.float(), b, c)):
        s = abip.Solver(*args, precision=precision, max_admm_iters=30)
        s.solve()
        states.append(s.state())
        s.close()
    assert np.array_equal(states[0], states[1]) and np.array_equal(states[0], states[2])


@pytest.mark.parametrize("which", [0, 1, 2])
def test_non_finite_device_input_is_refused(abip, which):
    lp = W.planted_dense(33, 71, seed=12)
    good = [torch.from_numpy(v).cuda() for v in (lp.A, lp.b, lp.c)]
    bad = [t.clone() for t in good]
    bad[which].view(-1)[-1] = float("inf")
    with pytest.raises(abip.AbipError) as e:
        abip.Solver(*bad)
    assert e.value.code == abip.ABIP_E_INVALID_ARG
    with pytest.raises(abip.AbipError) as e:
        abip.abip_solve_batch(*[list(p) for p in zip(good, bad)])
    assert e.value.code == abip.ABIP_E_INVALID_ARG


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_shared_batch_device_inputs_equal_host_inputs(abip, precision):
    """The shared-A batch reads a device A (FP32 or FP64), b and c in place: the bits of the host route."""
    lps = W.basis_pursuit(40, 90, batch=5, seed=21)
    prm = abip.default_params(precision=precision, max_admm_iters=40)
    A32 = lps.A.astype(np.float32)
    runs = []
    for A, on in ((lps.A, False), (torch.from_numpy(lps.A).cuda(), True), (torch.from_numpy(A32).cuda(), True)):
        vec = (lambda v: torch.from_numpy(v).cuda()) if on else (lambda v: v)
        infos, xs, ys, ss = abip.abip_solve_batch_shared(A, [vec(v) for v in lps.bs], [vec(v) for v in lps.cs], prm)
        runs.append(np.concatenate([np.concatenate(t) for t in (xs, ys, ss)]))
    assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])
    bad = [torch.from_numpy(v).cuda() for v in lps.bs]
    bad[3][-1] = float("nan")
    for A, b in ((torch.full((40, 180), float("inf"), device="cuda", dtype=torch.float64), lps.bs),
                 (torch.from_numpy(lps.A).cuda(), bad)):
        with pytest.raises(abip.AbipError) as e:
            abip.abip_solve_batch_shared(A, b, lps.cs, prm)
        assert e.value.code == abip.ABIP_E_INVALID_ARG


def test_shared_batch_waits_for_work_on_the_default_stream(abip):
    """A on the host; b and c on the device, written on the default stream after a long kernel."""
    lps = W.basis_pursuit(40, 90, batch=5, seed=22)
    prm = abip.default_params(max_admm_iters=20)
    want = np.concatenate(abip.abip_solve_batch_shared(lps.A, lps.bs, lps.cs, prm)[1])
    src = [torch.from_numpy(v).cuda() for v in [*lps.bs, *lps.cs]]
    dst = [torch.zeros_like(v) for v in src]
    busy = torch.ones(8192, 8192, device="cuda")
    torch.cuda.synchronize()
    for _ in range(20):   # some 10 ms each
        busy = busy @ busy * 1e-4
    for d, v in zip(dst, src):
        d.copy_(v)
    got = np.concatenate(abip.abip_solve_batch_shared(lps.A, dst[:5], dst[5:], prm)[1])
    assert np.array_equal(got, want)
