"""What a user of this package has it do, as timed cases: linear programs through every solver
path of the C ABI (dense, uneven batch, sparse PCG, sparse direct, batch sharing one matrix,
differentiable layer), from a 50 x 120 LP to the 100000 x 400000 one.

A case is a dict of plain values.  `kind` names the call:

  dense   one dense LP:  Solver(A, b, c).solve(), the handle released afterwards
  batch   `count` dense LPs of uneven size (m in [m_lo, m_hi], n = 2m .. 4m):  abip_solve_batch
  sparse  one CSR LP [R I] with 8 entries per column of R:  Solver + solve, or (`keep`) solve on
          a handle that the program set up before
  flow    min-cost flow on a side x side grid through the sparse LDL^T projection
  shared  `count` LPs with one dense A:  abip_solve_batch_shared; `lp` says which
          (basis pursuit, sparse inverse covariance columns, the paper's random LP)
  layer   `count` L1-SVM LPs through layer.lp_solve with gradients for A, b and c

ADMM needs 10^4 to 10^6 updates for a 1e-6 solve of most of these; `cap` bounds the updates of
one pass, so that a pass is a bounded piece of such a solve (status max_iter, the iterate is
returned as it stands).
"""
import math

import numpy as np
import torch

from paper_1805_12344_gb300 import abip, layer
from paper_1805_12344_gb300 import workloads as W

PRECISION = {"f64": abip.ABIP_PREC_F64, "mixed": abip.ABIP_PREC_MIXED, "bf16": abip.ABIP_PREC_MIXED_BF16}
F64 = torch.float64


def listed():
    return [
        # the smallest call: a small dense LP with the default parameters, towards the default 1e-6
        dict(name="dense_f64_50x120", kind="dense", lp="planted", m=50, n=120, precision="f64", cap=2000),
        # one L1-SVM at the size of the repository's config, default precision
        dict(name="dense_f64_svm", kind="dense", lp="svm", m=512, n=1154, precision="f64", cap=200),
        # the same LP as a user in a hurry runs it: FP64 state, FP32 products of changes
        dict(name="dense_mixed_svm", kind="dense", lp="svm", m=512, n=1154, precision="mixed", cap=800),
        # many unrelated small LPs at once (a service's queue), fewer than the GPU has SMs
        dict(name="batch_f64", kind="batch", count=64, m_lo=16, m_hi=256, precision="f64", cap=200),
        # the same recipe with more LPs than SMs, in mixed precision
        dict(name="batch_mixed", kind="batch", count=192, m_lo=16, m_hi=256, precision="mixed", cap=400),
        # one sparse LP of moderate size in the default precision (Jacobi-PCG projection)
        dict(name="sparse_f64", kind="sparse", m=2000, precision="f64", cg_tol=1e-10, cap=300, keep=False),
        # a small sparse LP in mixed precision: latency counts, the work is tiny
        dict(name="sparse_mixed_small", kind="sparse", m=300, precision="mixed", cg_tol=1e-10, cap=500, keep=False),
        # the headline workload: 100000 x 400000, 2.5 M entries, mixed precision, a kept handle
        # (a full solve is 10^5 updates and more, against one set-up)
        dict(name="sparse_mixed_large", kind="sparse", m=100000, precision="mixed", cg_tol=1e-8, cap=300, keep=True),
        # network flow through the sparse direct projection
        dict(name="flow_ldl", kind="flow", side=16, cap=400),
        # basis pursuit: one 2048 x 8192 dictionary, 64 measurements, products on the tensor cores
        dict(name="shared_bp_bf16", kind="shared", lp="bp", m=2048, n=16384, count=64, precision="bf16", cap=300),
        # sparse inverse covariance: 128 column LPs with one matrix, default precision
        dict(name="shared_sice_f64", kind="shared", lp="sice", m=256, n=512, count=128, precision="f64", cap=200),
        # a training step: 32 LPs forward, gradients of a loss on x* back to A, b and c
        dict(name="layer_svm", kind="layer", m=96, n=226, count=32, precision="f64", cap=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "batch", "sparse", "flow", "shared", "layer"])
    if kind == "dense":
        precision = rng.choice(["f64", "mixed"])
        m = _log(rng, 16, 512)
        if rng.random() < 0.5:
            return dict(kind=kind, lp="planted", m=m, n=int(m * rng.uniform(1.5, 4.0)), precision=precision,
                        cap=rng.randint(100, 400))
        m = max(m, 24)
        d = max(2, m // 8)
        return dict(kind=kind, lp="svm", m=m, n=2 * d + 2 + 2 * m, precision=precision, cap=rng.randint(100, 400))
    if kind == "batch":
        lo = _log(rng, 8, 128)
        return dict(kind=kind, count=_log(rng, 2, 256), m_lo=lo, m_hi=min(256, 2 * lo + rng.randint(0, 64)),
                    precision=rng.choice(["f64", "mixed"]), cap=rng.randint(50, 200))
    if kind == "sparse":
        m = _log(rng, 80, 60000)
        return dict(kind=kind, m=m, precision=rng.choice(["f64", "mixed"]), cg_tol=rng.choice([1e-8, 1e-10]),
                    cap=rng.randint(50, 300), keep=bool(m > 10000))
    if kind == "flow":
        return dict(kind=kind, side=_log(rng, 4, 40), cap=rng.randint(50, 200))
    if kind == "shared":
        lp = rng.choice(["bp", "sice", "random"])
        precision = rng.choice(["f64", "mixed", "bf16"])
        if lp == "bp":
            m = 128 * rng.randint(1, 6) if rng.random() < 0.5 else _log(rng, 24, 768)
            return dict(kind=kind, lp=lp, m=m, n=8 * m, count=_log(rng, 1, 64), precision=precision,
                        cap=rng.randint(50, 150))
        if lp == "sice":
            d = _log(rng, 16, 160)
            return dict(kind=kind, lp=lp, m=2 * d, n=4 * d, count=rng.randint(1, d), precision=precision,
                        cap=rng.randint(50, 200))
        m = _log(rng, 50, 500)
        return dict(kind=kind, lp=lp, m=m, n=int(m * rng.uniform(2, 10)), count=1, precision=precision,
                    cap=rng.randint(50, 300))
    m = 2 * _log(rng, 8, 64)
    return dict(kind=kind, m=m, n=2 * (m // 6) + 2 + 2 * m, count=_log(rng, 1, 64), precision=rng.choice(["f64", "mixed"]),
                cap=rng.randint(100, 500))


# --- inputs -------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape, dtype=F64):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=F64)


def _planted_pair(g, n, m):
    """x0: 30 % of the entries U[0.5, 2]; s0: U[0.5, 2] on the others; y0 ~ N(0, 1)."""
    on = torch.randperm(n, generator=g, device="cuda") < round(0.3 * n)
    v = _uniform(g, 0.5, 2.0, n)
    zero = torch.zeros_like(v)
    return torch.where(on, v, zero), _randn(g, m), torch.where(on, zero, v)


def _planted(g, m, n, twin=False):
    """A dense LP with a planted optimum, or (`twin`) its infeasible twin."""
    A = _randn(g, m, n, dtype=torch.float32).double()
    x0, y0, s0 = _planted_pair(g, n, m)
    b, c = A @ x0, A.T @ y0 + s0
    if twin:
        A[0] = _randn(g, n).abs().float().double()
        b[0] = -1.0
    return A, b, c


def _svm(g, m, n):
    """L1-SVM with m samples and d = (n - 2 - 2m) / 2 features: x = [w+, w-, b+, b-, xi, t]."""
    d = (n - 2 - 2 * m) // 2
    label = torch.ones(m, device="cuda", dtype=F64)
    label[torch.randperm(m, generator=g, device="cuda")[: m // 2]] = -1.0
    ya = label[:, None] * (_randn(g, m, d) + 0.5 * label[:, None])
    eye = torch.eye(m, device="cuda", dtype=F64)
    A = torch.cat([ya, -ya, label[:, None], -label[:, None], eye, -eye], 1).contiguous()
    c = torch.cat([torch.ones(2 * d, device="cuda", dtype=F64), torch.zeros(2, device="cuda", dtype=F64),
                   torch.ones(m, device="cuda", dtype=F64), torch.zeros(m, device="cuda", dtype=F64)])
    return A, torch.ones(m, device="cuda", dtype=F64), c


def _sizes(case):
    """The sizes of a batch's instances: a property of the case, not of the seed's values."""
    rng = np.random.default_rng([case["count"], case["m_lo"], case["m_hi"]])
    ms = rng.integers(case["m_lo"], case["m_hi"] + 1, size=case["count"])
    ns = np.round(ms * rng.uniform(2.0, 4.0, size=case["count"])).astype(int)
    twin = rng.random(case["count"]) < 0.1
    return [(int(m), int(n), bool(t)) for m, n, t in zip(ms, ns, twin)]


def _csr(rows, cols, vals, m, n):
    """workloads.CSR (host) of entries sorted by (row, column)."""
    order = torch.argsort(rows * n + cols, stable=True)
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return W.CSR(m=m, n=n, row_ptr=row_ptr.cpu().numpy(), col_idx=cols[order].int().cpu().numpy(),
                 val=vals[order].float().cpu().numpy())


def _csr_times(A, x):
    """A x on the host, row by row in a fixed order (no row of these matrices is empty)."""
    return np.add.reduceat(A.val.astype(np.float64) * x[A.col_idx], A.row_ptr[:-1])


def _sparse_lp(seed, m):
    """A = [R I], R m x 3m with 8 entries N(0, 1) (float32) per column at distinct rows."""
    g = _gen(seed)
    nr, per = 3 * m, min(8, m)
    rows = torch.randint(0, m, (nr, per), generator=g, device="cuda")
    while True:
        srt = rows.sort(1).values
        bad = (srt[:, 1:] == srt[:, :-1]).any(1).nonzero()[:, 0]
        if bad.numel() == 0:
            break
        rows[bad] = torch.randint(0, m, (bad.numel(), per), generator=g, device="cuda")
    vals = _randn(g, nr, per, dtype=torch.float32)
    cols = torch.arange(nr, device="cuda")[:, None].expand(nr, per)
    eye = torch.arange(m, device="cuda")
    n = nr + m
    A = _csr(torch.cat([rows.reshape(-1), eye]), torch.cat([cols.reshape(-1), nr + eye]),
             torch.cat([vals.reshape(-1), torch.ones(m, device="cuda")]), m, n)
    x0, y0, s0 = _planted_pair(g, n, m)
    aty = torch.cat([(vals.double() * y0[rows]).sum(1), y0])
    return A, _csr_times(A, x0.cpu().numpy()), (aty + s0).cpu().numpy()


def _flow_lp(seed, side):
    """The repository's grid flow LP: +1 where an arc leaves a node, -1 where it enters."""
    lp = W.grid_flow(side, seed=int(seed))
    return lp.A, lp.b, lp.c


def _shared_lp(seed, case):
    """(A, bs, cs): one matrix, `count` right-hand sides and costs, as rows of two tensors."""
    g = _gen(seed)
    m, n, B = case["m"], case["n"], case["count"]
    if case["lp"] == "bp":        # A = [D, -D], b_k = D x_k with 5 % nonzeros, c = e
        nd = n // 2
        D = (_randn(g, m, nd) / math.sqrt(m)).float().double()
        A = torch.cat([D, -D], 1).contiguous()
        xt = _randn(g, B, nd) * (torch.rand(B, nd, generator=g, device="cuda") < 0.05)
        return A, xt @ D.T, torch.ones(B, n, device="cuda", dtype=F64)
    if case["lp"] == "sice":      # columns of sparse inverse covariance, bounds as slack rows
        d = m // 2
        X = _randn(g, 2 * d, d)
        X = X + 0.4 * X.roll(1, 1)
        S = X.T @ X / (2 * d)
        S = S / S.diagonal().max()
        lam = 1.5 * math.sqrt(math.log(max(d, 2)) / (2 * d))
        eye, zero = torch.eye(d, device="cuda", dtype=F64), torch.zeros(d, d, device="cuda", dtype=F64)
        # S (b+ - b-) - r = e_j - lam e,  r + t = 2 lam e
        A = torch.cat([torch.cat([S, -S, -eye, zero], 1), torch.cat([zero, zero, eye, eye], 1)]).contiguous()
        b = torch.full((B, m), 2 * lam, device="cuda", dtype=F64)
        b[:, :d] = eye[torch.arange(B, device="cuda") % d] - lam
        c = torch.zeros(B, n, device="cuda", dtype=F64)
        c[:, : 2 * d] = 1.0
        return A, b, c
    # the paper's random LP: A = U^T D V, U and V of density 0.2
    U = _randn(g, m, m) * (torch.rand(m, m, generator=g, device="cuda") < 0.2)
    V = _randn(g, m, n) * (torch.rand(m, n, generator=g, device="cuda") < 0.2)
    A = (U.T @ (_randn(g, m)[:, None] * V)).contiguous()
    b, c = [], []
    for _ in range(B):
        k = torch.rand(n, generator=g, device="cuda")
        v = _randn(g, n).abs()
        x0 = torch.where(k < 0.6, torch.zeros_like(v), torch.where(k < 0.7, 10 * v, 0.1 * v))
        b.append(A @ x0)
        c.append(A.T @ _randn(g, m) + torch.where(k < 0.6, v, torch.zeros_like(v)))
    return A, torch.stack(b), torch.stack(c)


def _params(case):
    p = dict(max_admm_iters=case["cap"])
    if "precision" in case:
        p["precision"] = PRECISION[case["precision"]]
    if "cg_tol" in case:
        p["cg_tol"] = case["cg_tol"]
    return p


def _one_lp(case, seed):
    g = _gen(seed)
    return (_planted if case["lp"] == "planted" else _svm)(g, case["m"], case["n"])


def _layer_lp(case, seed):
    g = _gen(seed)
    A, b, c = (torch.stack(t) for t in zip(*[_svm(g, case["m"], case["n"]) for _ in range(case["count"])]))
    return A, b, c + 0.1 * torch.rand(c.shape, generator=g, device="cuda", dtype=F64), _randn(g, *c.shape)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, params=_params(case))
    if kind == "dense":
        st["lp"] = _one_lp(case, seed)
    elif kind == "batch":
        g = _gen(seed)
        st["lp"] = list(zip(*[_planted(g, m, n, t) for m, n, t in _sizes(case)]))
        st["prm"] = abip.default_params(**st["params"])
    elif kind == "sparse":
        st["lp"] = _sparse_lp(seed, case["m"])
        if case["keep"]:
            st["solver"] = abip.Solver(*st["lp"], **st["params"])
    elif kind == "flow":
        st["lp"] = _flow_lp(seed, case["side"])
        st["params"]["linsys"] = abip.ABIP_LINSYS_SPARSE_LDL
    elif kind == "shared":
        st["lp"] = _shared_lp(seed, case)
        st["prm"] = abip.default_params(**st["params"])
    else:
        st["lp"] = _layer_lp(case, seed)
    return st


# --- one pass -----------------------------------------------------------------------------

def _answer(infos, x, y, s):
    return dict(x=x, y=y, s=s, obj=torch.tensor([f["obj"] for f in infos], dtype=F64),
                status=torch.tensor([f["status"] for f in infos]), updates=torch.tensor([f["admm_iters"] for f in infos]))


def run(state):
    kind, lp = state["case"]["kind"], state["lp"]
    if kind in ("dense", "flow", "sparse"):
        solver = state.get("solver") or abip.Solver(*lp, **state["params"])
        info, x, y, s = solver.solve(device_out=kind == "dense")
        if "solver" not in state:
            solver.close()
        return _answer([info], x, y, s)
    if kind == "batch":
        infos, xs, ys, ss = abip.abip_solve_batch(*lp, state["prm"], device_out=True)
        return _answer(infos, torch.cat(xs), torch.cat(ys), torch.cat(ss))
    if kind == "shared":
        A, b, c = lp
        infos, xs, ys, ss = abip.abip_solve_batch_shared(A, list(b), list(c), state["prm"], device_out=True)
        return _answer(infos, torch.stack(xs), torch.stack(ys), torch.stack(ss))
    A, b, c, target = lp
    A, b, c = (t.detach().requires_grad_() for t in (A, b, c))
    x = layer.lp_solve(A, b, c, eps=1e-3, **state["params"])
    dA, db, dc = torch.autograd.grad(((x - target) ** 2).sum(), (A, b, c))
    return dict(x=x.detach(), dA=dA, db=db, dc=dc)


def work(case):
    """Inputs read once, outputs written once; per ADMM update the products that the projection and
    the tests cannot do without (one with A, one with A^T, one solve with the factor or the PCG
    iterations it takes at least) and about 40 operations per column."""
    kind, cap = case["kind"], case["cap"]

    def dense(m, n, nb=1, shared=False):
        data = 8.0 * ((1 if shared else nb) * m * n + nb * (m + n + 2 * n + m))
        setup = (1 if shared else nb) * (m * m * n + m ** 3 / 3.0)
        return data, setup + nb * cap * (4.0 * m * n + 2.0 * m * m + 40.0 * (m + n))

    if kind == "dense":
        by, fl = dense(case["m"], case["n"])
    elif kind == "batch":
        by, fl = (sum(t) for t in zip(*[dense(m, n) for m, n, _ in _sizes(case)]))
    elif kind == "shared":
        by, fl = dense(case["m"], case["n"], case["count"], True)
    elif kind == "sparse":
        m, n = case["m"], 4 * case["m"]
        nnz = 25.0 * m
        by = nnz * 8 + 8.0 * (m + n + 2 * n + m)
        fl = cap * (5 * 4 * nnz + 4 * nnz + 40.0 * (m + n))
    elif kind == "flow":
        m, n = case["side"] ** 2 - 1, 4 * case["side"] * (case["side"] - 1)
        by = 2.0 * n * 8 + 8.0 * (m + n + 2 * n + m)
        fl = cap * (4 * 2.0 * n + 4 * 4.0 * n + 40.0 * (m + n))
    else:
        m, n, nb = case["m"], case["n"], case["count"]
        by, fl = dense(m, n, nb)
        by += nb * 8.0 * (m * n + m + n + n)
        fl += nb * (m * m * n + m ** 3 / 3.0 + 4.0 * m * n)
    return dict(bytes=by, flops=fl)


# --- the same in 64 bits with plain torch -------------------------------------------------

class _Dense:
    """A batch of dense LPs padded to one size: A [B or 1, m, n], masks of the real rows and columns."""

    def __init__(self, A):
        self.A, self.AT = A, A.transpose(-1, -2)
        G = torch.eye(A.shape[1], device="cuda", dtype=F64) + A @ self.AT
        self.L = torch.linalg.cholesky(G)
        self.Ginv = torch.cholesky_inverse(self.L)

    def mul(self, x):
        return (x @ self.AT[0]) if self.A.shape[0] == 1 else torch.einsum("bij,bj->bi", self.A, x)

    def tmul(self, y):
        return (y @ self.A[0]) if self.A.shape[0] == 1 else torch.einsum("bij,bi->bj", self.A, y)

    def solve(self, q):
        return (q @ self.Ginv[0]) if self.A.shape[0] == 1 else torch.einsum("bij,bj->bi", self.Ginv, q)


class _Sparse:
    """One sparse LP; G^{-1} by Jacobi-preconditioned conjugate gradients to 1e-14."""

    def __init__(self, A):
        rp, ci = torch.from_numpy(A.row_ptr).cuda(), torch.from_numpy(A.col_idx.astype(np.int64)).cuda()
        v = torch.from_numpy(A.val.astype(np.float64)).cuda()
        rows = torch.repeat_interleave(torch.arange(A.m, device="cuda"), rp[1:] - rp[:-1])
        order = torch.argsort(ci * A.m + rows)
        cp = torch.zeros(A.n + 1, dtype=torch.int64, device="cuda")
        cp[1:] = torch.cumsum(torch.bincount(ci, minlength=A.n), 0)
        self.A = torch.sparse_csr_tensor(rp, ci, v, (A.m, A.n))
        self.AT = torch.sparse_csr_tensor(cp, rows[order], v[order], (A.n, A.m))
        self.d = 1.0 / (1.0 + torch.zeros(A.m, device="cuda", dtype=F64).index_add_(0, rows, v * v))
        self.z = None

    def mul(self, x):
        return (self.A @ x[0])[None]

    def tmul(self, y):
        return (self.AT @ y[0])[None]

    def solve(self, q):
        z = torch.zeros_like(q) if self.z is None else self.z.clone()
        r = q - z - self.mul(self.tmul(z))
        p = self.d * r
        rz = (r * p).sum()
        stop = 1e-14 * max(1.0, float(q.norm()))
        for k in range(400):
            if k % 6 == 0 and float(r.norm()) <= stop:
                break
            gp = p + self.mul(self.tmul(p))
            a = rz / (p * gp).sum()
            z = z + a * p
            r = r - a * gp
            zr = self.d * r
            new = (r * zr).sum()
            p = zr + (new / rz) * p
            rz = new
        self.z = z
        return z


def _admm(op, b, c, rows, cols, cap, eps=1e-6, alpha=1.8, gamma=0.1):
    """ABIP for the rows of b [B, m], c [B, n] (masks `rows`, `cols`): the paper's Algorithm 2 with
    over-relaxation on the self-dual embedding, beta = 1.  Returns the state, a dict."""
    B, dev = b.shape[0], "cuda"
    one = cols.to(F64)
    bbar, cbar = b - op.mul(one), c - one
    zbar, xi = c.sum(1) + 1.0, -cols.sum(1).to(F64) - 1.0
    nb, nc = b.norm(dim=1), c.norm(dim=1)

    def proj(a, d):
        zy = op.solve(a - op.mul(d))
        return zy, d + op.tmul(zy)

    g1y, g1x = proj(-b, c)
    g2y, g2x = proj(bbar, -cbar)

    def ht(zy, zx):
        return (c * zx).sum(1) - (b * zy).sum(1), (bbar * zy).sum(1) - (cbar * zx).sum(1)

    k00, k10 = ht(g1y, g1x)
    k01, k11 = ht(g2y, g2x)
    k00, k01, k10, k11 = 1 + k00, zbar + k01, k10 - zbar, 1 + k11
    det = k00 * k11 - k01 * k10

    def prox(w, t):
        D = (w * w + 4 * t).sqrt()
        big, small = 0.5 * (w.abs() + D), 2 * t / (w.abs() + D)
        return torch.where(w >= 0, big, small), torch.where(w >= 0, small, big)

    y = torch.zeros_like(b)
    x, s = one.clone(), one.clone()
    tau, kappa, theta, mu = (torch.ones(B, device=dev, dtype=F64) for _ in range(4))
    total, status = (torch.zeros(B, device=dev, dtype=torch.int64) for _ in range(2))
    stepped = torch.zeros(B, device=dev, dtype=torch.bool)
    v = lambda t: t[:, None]  # noqa: E731
    for cycle in range(cap + 64):
        Ax, As, aty = op.mul(x), op.mul(s), op.tmul(y)
        ry = Ax - b * v(tau) + bbar * v(theta)
        rx = (-aty + c * v(tau) - cbar * v(theta) - s) * one
        bty, ctx = (b * y).sum(1), (c * x).sum(1)
        rt = bty - ctx + zbar * theta - kappa
        rth = -(bbar * y).sum(1) + (cbar * x).sum(1) - zbar * tau - xi
        inner = (ry * ry).sum(1) + (rx * rx).sum(1) + rt * rt + rth * rth
        dual = (aty + s) * one
        pres = (Ax / v(tau) - b).norm(dim=1) / (1 + nb)
        dres = (dual / v(tau) - c).norm(dim=1) / (1 + nc)
        gap = (ctx / tau - bty / tau).abs() / (1 + (ctx / tau).abs() + (bty / tau).abs())
        now = torch.zeros_like(status)
        now[(ctx < 0) & (Ax.norm(dim=1) <= eps * -ctx / nc)] = abip.ABIP_DUAL_INFEASIBLE
        now[(bty > 0) & (dual.norm(dim=1) <= eps * bty / nb)] = abip.ABIP_PRIMAL_INFEASIBLE
        now[(pres <= eps) & (dres <= eps) & (gap <= eps)] = abip.ABIP_OPTIMAL
        now = torch.where((now == 0) & (total >= cap), torch.full_like(now, abip.ABIP_MAX_ITER), now)
        status = torch.where((status == 0) & stepped, now, status)
        live = status == 0
        if cycle % 16 == 0 and not bool(live.any()):
            break
        warm = live & (inner <= mu)
        step = live & ~warm
        # the update, for the instances that take one
        zy = op.solve(y - Ax - As)
        zx = (x + s) + op.tmul(zy)
        h0, h1 = ht(zy, zx)
        v1, v2 = tau + kappa + h0, theta + xi + h1
        t1, t2 = (k11 * v1 - k01 * v2) / det, (k00 * v2 - k10 * v1) / det
        uy = zy - g1y * v(t1) - g2y * v(t2)
        ux = zx - g1x * v(t1) - g2x * v(t2)
        yn = alpha * uy + (1 - alpha) * y
        xn, sn = prox(alpha * ux + (1 - alpha) * x - s, v(mu))
        tn, kn = prox(alpha * t1 + (1 - alpha) * tau - kappa, mu)
        thn = alpha * t2 + (1 - alpha) * theta
        # the warm start, for those whose inner loop has ended
        keep = x >= s
        xw, sw = torch.where(keep, x, gamma * x), torch.where(keep, gamma * s, s)
        tw, kw = torch.where(tau >= kappa, tau, gamma * tau), torch.where(tau >= kappa, gamma * kappa, kappa)
        root = math.sqrt(gamma)

        def pick(old, new, ws):
            a, w = (step, warm) if old.dim() == 1 else (v(step), v(warm))
            return torch.where(a, new, torch.where(w, ws, old))

        y, x, s = pick(y, yn, root * y), pick(x, xn, xw) * one, pick(s, sn, sw) * one
        tau, kappa, theta = pick(tau, tn, tw), pick(kappa, kn, kw), pick(theta, thn, root * theta)
        mu = torch.where(warm, gamma * mu, mu)
        total = total + step.long()
        stepped = step
    return dict(x=x, y=y, s=s, tau=tau, kappa=kappa, theta=theta, mu=mu, status=status, bty=bty, ctx=ctx,
                bbar=bbar, cbar=cbar, zbar=zbar)


def _scaled(r):
    sx, sy = 1 / r["tau"], 1 / r["tau"]
    pinf, dinf = r["status"] == abip.ABIP_PRIMAL_INFEASIBLE, r["status"] == abip.ABIP_DUAL_INFEASIBLE
    sx = torch.where(pinf, torch.ones_like(sx), torch.where(dinf, -1 / r["ctx"], sx))
    sy = torch.where(pinf, 1 / r["bty"], torch.where(dinf, torch.ones_like(sy), sy))
    return r["x"] * sx[:, None], r["y"] * sy[:, None], r["s"] * sy[:, None]


def _all(b, c):
    return torch.ones_like(b, dtype=torch.bool), torch.ones_like(c, dtype=torch.bool)


def _gradient(A, b, c, r, g):
    """dL/d(A, b, c) at the central point of the embedding that the iterate approximates, from
    g = dL/dx* (x* = x / tau): Newton onto the point, then the adjoint of its Jacobian."""
    m, n = A.shape
    y, x, s = r["y"].clone(), r["x"].clone(), r["s"].clone()
    tau, kappa, theta, mu = (r[k].clone() for k in ("tau", "kappa", "theta", "mu"))
    bbar, cbar, zbar = r["bbar"], r["cbar"], r["zbar"]
    N, xi = m + n + 2, -n - 1.0
    Q = torch.zeros(N, N, device="cuda", dtype=F64)
    Q[:m, m:m + n], Q[m:m + n, :m] = A, -A.T
    Q[:m, -2], Q[-2, :m], Q[:m, -1], Q[-1, :m] = -b, b, bbar, -bbar
    Q[m:-2, -2], Q[-2, m:-2], Q[m:-2, -1], Q[-1, m:-2] = c, -c, -cbar, cbar
    Q[-2, -1], Q[-1, -2] = zbar, -zbar

    def jac():
        d = torch.zeros(N, device="cuda", dtype=F64)
        d[m:m + n] = s / x
        d[-2] = kappa / tau
        return Q + torch.diag(d)

    best = None
    for _ in range(60):
        u = torch.cat([y, x, tau[None], theta[None]])
        F = Q @ u
        F[m:m + n] -= s
        F[-2] -= kappa
        F[-1] -= xi
        f5, f6 = x * s - mu, tau * kappa - mu
        size = float((F @ F + f5 @ f5 + f6 * f6).sqrt())
        if best is not None and size > 0.5 * best and size < 1e-10:
            break
        best = size if best is None else min(best, size)
        rhs = -F
        rhs[m:m + n] -= f5 / x
        rhs[-2] -= f6 / tau
        K = jac()
        d = torch.linalg.solve(K, rhs)
        d = d + torch.linalg.solve(K, rhs - K @ d)
        dx, dt = d[m:m + n], d[-2]
        ds, dk = (-f5 - s * dx) / x, (-f6 - kappa * dt) / tau
        at, by = torch.cat([x, s, tau[None], kappa[None]]), torch.cat([dx, ds, dt[None], dk[None]])
        a = min(1.0, float(torch.where(by < 0, -0.99 * at / by, torch.full_like(at, math.inf)).min()))
        y, x, s = y + a * d[:m], x + a * dx, s + a * ds
        tau, theta, kappa = tau + a * dt, theta + a * d[-1], kappa + a * dk
    rhs = torch.zeros(N, device="cuda", dtype=F64)
    rhs[m:m + n] = g / tau
    rhs[-2] = -(g @ x) / (tau * tau)
    KT = jac().T.contiguous()
    lam = torch.linalg.solve(KT, rhs)
    lam = lam + torch.linalg.solve(KT, rhs - KT @ lam)
    l1, l2, l3, l4 = lam[:m], lam[m:m + n], lam[-2], lam[-1]
    db = -(l1 * (theta - tau) + (l3 - l4) * y)
    dc = -(l2 * (tau - theta) + l3 * (theta - x) + l4 * (x - tau))
    dA = -(l1[:, None] * (x - theta)[None] - y[:, None] * l2[None] + l4 * y[:, None])
    return dA, db, dc


def exact(case, seed):
    kind, cap = case["kind"], case["cap"]
    if kind == "layer":
        A, b, c, target = _layer_lp(case, seed)
        r = _admm(_Dense(A), b, c, *_all(b, c), cap, eps=1e-3)
        x, _, _ = _scaled(r)
        grads = [_gradient(A[k], b[k], c[k], {q: t[k] for q, t in r.items()}, 2 * (x[k] - target[k]))
                 for k in range(case["count"])]
        dA, db, dc = (torch.stack(t) for t in zip(*grads))
        return dict(x=x, dA=dA, db=db, dc=dc)
    if kind == "batch":
        g = _gen(seed)
        lps = [_planted(g, m, n, t) for m, n, t in _sizes(case)]
        m, n, B = max(l[0].shape[0] for l in lps), max(l[0].shape[1] for l in lps), len(lps)
        A, b, c = (torch.zeros(B, *d, device="cuda", dtype=F64) for d in ((m, n), (m,), (n,)))
        rows, cols = torch.zeros_like(b, dtype=torch.bool), torch.zeros_like(c, dtype=torch.bool)
        for k, (a, bb, cc) in enumerate(lps):
            A[k, : a.shape[0], : a.shape[1]], b[k, : bb.numel()], c[k, : cc.numel()] = a, bb, cc
            rows[k, : bb.numel()], cols[k, : cc.numel()] = True, True
        r = _admm(_Dense(A), b, c, rows, cols, cap)
        x, y, s = _scaled(r)
        return dict(x=x[cols], y=y[rows], s=s[cols], obj=(r["ctx"] / r["tau"]).cpu(), status=None, updates=None)
    if kind == "sparse":
        A, b, c = _sparse_lp(seed, case["m"])
    elif kind == "flow":
        A, b, c = _flow_lp(seed, case["side"])
    elif kind == "shared":
        A, b, c = _shared_lp(seed, case)
    else:
        A, b, c = _one_lp(case, seed)
    if kind in ("sparse", "flow"):
        b, c = torch.from_numpy(b).cuda(), torch.from_numpy(c).cuda()
        op = _Sparse(A) if A.m * A.n > 4_000_000 else _Dense(torch.from_numpy(A.to_dense()).cuda()[None])
    else:
        op = _Dense(A[None])
    if kind != "shared":
        b, c = b[None], c[None]
    r = _admm(op, b, c, *_all(b, c), cap)
    x, y, s = _scaled(r)
    obj = (r["ctx"] / r["tau"]).cpu()
    if kind == "shared":
        return dict(x=x, y=y, s=s, obj=obj, status=None, updates=None)
    x, y, s = (t[0] if kind == "dense" else t[0].cpu().numpy() for t in (x, y, s))
    return dict(x=x, y=y, s=s, obj=obj, status=None, updates=None)
