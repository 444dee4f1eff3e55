"""The autotuner's choice is kept per kernel: one timed on the cluster kernels is not served to the
one-CTA kernel (Barzilai-Borwein batches), nor is a file's entry that does not name its kernel."""
import json
import os
import subprocess
import sys

import pytest

from paper_1805_12344_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def abip():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1805_12344_gb300 import build, abip as _abip
    build.build()
    _abip.lib()
    return _abip


def test_each_kernel_is_timed(abip):
    lps = W.batch_uneven(count=10, infeasible_frac=0.0, m_lo=16, m_hi=40, seed=17)
    args = ([l.A for l in lps], [l.b for l in lps], [l.c for l in lps])
    for want in (1, 2):
        for bb in (0, 1):
            infos, *_ = abip.abip_solve_batch(*args, abip.default_params(autotune=1, bb_beta=bb, max_admm_iters=200))
            assert infos[0]["tuned"] == want, (want, bb)


def test_a_files_entry_without_its_kernel_is_not_used(abip, tmp_path):
    cache = tmp_path / "tune.json"
    lps = W.batch_uneven(count=12, infeasible_frac=0.0, m_lo=16, m_hi=32, seed=5)
    mn = sum(float(l.A.shape[0] * l.A.shape[1]) for l in lps)
    old = f"{torch.cuda.get_device_name(0)}|f64|count=12|mmax={max(l.A.shape[0] for l in lps)}|mn={mn:.1e}".replace(":", "_")
    cache.write_text('{\n  "%s": 2\n}\n' % old)
    code = ("import sys; sys.path.insert(0, %r)\n"
            "from paper_1805_12344_gb300 import abip, workloads as W\n"
            "lps = W.batch_uneven(count=12, infeasible_frac=0.0, m_lo=16, m_hi=32, seed=5)\n"
            "infos, *_ = abip.abip_solve_batch([l.A for l in lps], [l.b for l in lps], [l.c for l in lps],\n"
            "                                   abip.default_params(autotune=1, max_admm_iters=200), want_solution=False)\n"
            "print('TUNED', infos[0]['tuned'])\n") % ROOT
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, ABIP_TUNE_CACHE=str(cache)), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    assert "TUNED 1" in r.stdout
    entries = json.loads(cache.read_text())
    assert entries[old] == 2 and len(entries) == 2   # the file's own entry stays
