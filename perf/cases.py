"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` gives the standing ones, ``draw(rng)`` one more
of the same ranges; ``prepare(case, seed)`` makes what a program has in hand before the call,
``run(state)`` is one pass through the public entry points, ``work(case)`` the bytes and
operations that the pass cannot do without, and ``exact(case, seed)`` its outputs as plain
torch gives them in 64 bits.

Sizes: the CI-like workload of bench.py (n up to 2,000,000, k = 16 and 5 extra vectors, so
blocks of 21 columns and bases of 63), the cfg1 workload (n = 4096, k = 4), the dense
CASSCF-like workload (n = 8192, k = 8 and 5 extra), and odd and ragged sizes between them.
"""
from __future__ import annotations

import math

import torch

import paper_2305_06668_gb300 as lb


def listed():
    return [
        # Algorithm 2 on the first block of the n = 4096 workload: the smallest call, launches and latency
        dict(name="ortho_cfg1", kind="ortho", n=4096, p=4, q=0),
        # Algorithm 3 in a plain FP64 solve of mid size: W against (X, P) once k = 16 pairs iterate
        dict(name="ortho_against", kind="ortho", n=300_007, p=21, q=42),
        # Rayleigh-Ritz matrix V^T AV of a plain FP64 solve, m = 21, s = 63
        dict(name="gram_rr_f64", kind="gram", n=1_000_000, p=63, q=63, arith="f64"),
        # the same of the mixed form's FP32 phase on the largest workload (tensor cores)
        dict(name="gram_rr_f32", kind="gram", n=2_000_000, p=63, q=63, arith="f32"),
        # X, AX = (V, AV) u_x with the residual norms: FP32 phase, largest workload
        dict(name="update_rr_f32", kind="update", n=2_000_000, w=21, q=21, arith="f32", pair=True),
        # the same of the FP64 refinement of a mixed solve
        dict(name="update_rr_f64", kind="update", n=1_000_000, w=21, q=21, arith="f64", pair=True),
        # A W of a plain FP64 solve on a CI-like matrix, k = 16
        dict(name="spmm_ci_f64", kind="spmm", n=500_000, p=16, arith="f64"),
        # A W of the dense orbital-Hessian workload, k = 8 and 5 extra
        dict(name="spmm_dense", kind="dense", n=8192, p=13),
        # Rayleigh-Ritz eigensolve of a basis of 63 vectors
        dict(name="syev_rr", kind="syev", s=63, two_stage=False),
        # the tridiagonal preconditioner on a block of residuals of a mid-sized problem
        dict(name="precond_tridiag", kind="tridiag", n=100_000, p=21),
        # a whole plain FP64 solve of the n = 4096 workload (default options)
        dict(name="solve_cfg1_f64", kind="solve", form="f64", n=4096, k=4, extra=0, tol=1e-12),
        # a whole solve in the headline form: mixed precision, learned preconditioner
        dict(name="solve_ci_mixed", kind="solve", form="mixed", n=2_000_000, k=16, extra=5, tol=1e-8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ortho", "gram", "gram", "update", "update", "spmm", "dense", "syev", "tridiag", "solve"])
    if kind == "ortho":
        n, p = _log(rng, 2000, 1_000_000), rng.randint(1, 32)
        return dict(kind=kind, n=n, p=p, q=rng.choice([0, p, 2 * p, rng.randint(1, 64)]))
    if kind == "gram":
        # V^T AV, Y^T W and W^T W of every phase
        p = rng.randint(1, 96)
        q = rng.choice([p, (p + 1) // 2, rng.randint(1, 96)])
        return dict(kind=kind, n=_log(rng, 2000, 1_500_000), p=p, q=q, arith=rng.choice(["f64", "f64", "df", "f32"]))
    if kind == "update":
        w = rng.randint(1, 32)
        return dict(kind=kind, n=_log(rng, 2000, 1_500_000), w=w, q=rng.randint(1, w),
                    arith=rng.choice(["f32", "f64"]), pair=rng.choice([True, False]))
    if kind == "spmm":
        return dict(kind=kind, n=_log(rng, 4000, 700_000), p=rng.randint(1, 32), arith=rng.choice(["f64", "df"]))
    if kind == "dense":
        return dict(kind=kind, n=_log(rng, 300, 12_000), p=rng.randint(1, 32))
    if kind == "syev":
        return dict(kind=kind, s=rng.randint(3, 96), two_stage=rng.choice([True, False]))
    if kind == "tridiag":
        return dict(kind=kind, n=_log(rng, 2000, 500_000), p=rng.randint(1, 32))
    if rng.choice([True, False]):
        return dict(kind="solve", form="f64", n=_log(rng, 2000, 60_000), k=rng.randint(2, 16), extra=rng.randint(0, 5),
                    tol=1e-12)
    return dict(kind="solve", form="mixed", n=_log(rng, 50_000, 1_000_000), k=rng.randint(4, 16), extra=5, tol=1e-8)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _block(g, n, w, dtype=torch.float64, ld=None):
    """Row-major n x w block of N(0, 1) entries, its rows padded to whole 16-byte units as the
    solver lays its blocks out."""
    vec = 4 if dtype == torch.float32 else 2
    ld = (w + vec - 1) // vec * vec if ld is None else ld
    buf = torch.zeros((n, ld), dtype=dtype, device="cuda")
    buf[:, :w] = torch.randn((n, w), generator=g, dtype=dtype, device="cuda")
    return buf[:, :w]


def _csr(i, j, v, diag):
    """Symmetric CSR from strict upper-triangle triplets (i < j, repeated pairs keep the first)."""
    n = diag.numel()
    key = i * n + j
    sk, perm = torch.sort(key, stable=True)
    first = torch.ones_like(sk, dtype=torch.bool)
    first[1:] = sk[1:] != sk[:-1]
    keep = perm[first]
    i, j, v = i[keep], j[keep], v[keep]
    del key, sk, perm, first, keep
    ar = torch.arange(n, device="cuda", dtype=torch.int64)
    rows, cols, vals = torch.cat([i, j, ar]), torch.cat([j, i, ar]), torch.cat([v, v, diag])
    del i, j, v
    order = torch.argsort(rows * n + cols)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return dict(row_ptr=row_ptr, col_idx=cols[order].to(torch.int32), val=vals[order], diag=diag)


def _ci(n, seed):
    """CI-like matrix: diagonal 0.001 i + U(0, 0.01), per row 28 couplings inside (i, i + 256]
    and 4 anywhere above, mirrored, N(0, 0.005^2)."""
    g = _gen(seed)
    ar = torch.arange(n, device="cuda", dtype=torch.int64)
    diag = 0.001 * ar.double() + 0.01 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    off = torch.empty((n, 28), dtype=torch.int64, device="cuda")
    for r in range(0, n, 1 << 19):
        m = min(1 << 19, n - r)
        off[r:r + m] = torch.rand((m, 256), generator=g, device="cuda").topk(28, dim=1).indices + 1
    far = 1 + (torch.rand((n, 4), generator=g, device="cuda", dtype=torch.float64)
               * (n - 1 - ar)[:, None].clamp(min=1)).long()
    i = ar[:, None].expand(n, 32).reshape(-1)
    j = (ar[:, None] + torch.cat([off, far], 1)).reshape(-1)
    ok = j < n
    i, j = i[ok], j[ok]
    v = 0.005 * torch.randn(i.numel(), generator=g, device="cuda", dtype=torch.float64)
    return _csr(i, j, v, diag)


def _cfg1(n, seed):
    """Diagonally dominant matrix: sorted diagonal 0.01 i + U(0, 0.005), 16 random couplings per
    row, mirrored, N(0, 0.01^2)."""
    g = _gen(seed)
    ar = torch.arange(n, device="cuda", dtype=torch.int64)
    diag = torch.sort(0.01 * ar.double() + 0.005 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).values
    i = ar.repeat_interleave(16)
    r = torch.randint(0, n - 1, (16 * n,), generator=g, device="cuda")
    j = torch.where(r >= i, r + 1, r)
    v = 0.01 * torch.randn(16 * n, generator=g, device="cuda", dtype=torch.float64)
    return _csr(torch.minimum(i, j), torch.maximum(i, j), v, diag)


def _guess(diag, m):
    """Unit vectors at the m smallest diagonal entries."""
    x = torch.zeros((diag.numel(), m), dtype=torch.float64, device="cuda")
    x[torch.argsort(diag, stable=True)[:m], torch.arange(m, device="cuda")] = 1.0
    return x


def prepare(case, seed):
    c, g = dict(case), _gen(seed)
    kind = c["kind"]
    s = dict(case=c)
    if kind == "ortho":
        n, p, q = c["n"], c["p"], c["q"]
        # columns of different length with some overlap, as preconditioned residuals have
        s["W0"] = _block(g, n, p)
        mix = torch.eye(p, dtype=torch.float64, device="cuda") + 0.2 * torch.rand((p, p), generator=g, dtype=torch.float64,
                                                                                  device="cuda") / p
        s["W0"].copy_(s["W0"] @ mix * torch.logspace(-3, 0, p, dtype=torch.float64, device="cuda"))
        s["W"] = _block(g, n, p)
        s["Y"] = None
        if q:
            s["Y"] = _block(g, n, q)
            # the orthonormal (X, P) that the iteration holds
            s["Y"].copy_(torch.linalg.qr(s["Y"].contiguous()).Q)
    elif kind == "gram":
        dt = torch.float32 if c["arith"] == "f32" else torch.float64
        vec = 4 if dt == torch.float32 else 2
        ld = (max(c["p"], c["q"]) + vec - 1) // vec * vec
        s["X"], s["Y"] = _block(g, c["n"], c["p"], dt, ld), _block(g, c["n"], c["q"], dt, ld)
    elif kind == "update":
        dt = torch.float32 if c["arith"] == "f32" else torch.float64
        n, w, q = c["n"], c["w"], c["q"]
        s["V"] = [_block(g, n, w, dt) for _ in range(3)]
        # Ritz coefficients: orthonormal columns
        s["U"] = torch.linalg.qr(torch.randn((3 * w, 3 * w), generator=g, dtype=torch.float64, device="cuda")).Q[:, :q]
        s["U"] = s["U"].t().contiguous().t()
        if c["pair"]:
            s["AV"] = [_block(g, n, w, dt) for _ in range(3)]
            s["lam"] = torch.linspace(0.003, 0.02, q, dtype=torch.float64, device="cuda")
    elif kind == "spmm":
        s["A"] = _ci(c["n"], seed)
        s["X"], s["Y"] = _block(g, c["n"], c["p"]), _block(g, c["n"], c["p"])
    elif kind == "dense":
        n, r = c["n"], max(1, c["n"] // 32)
        # D + U S U^T: D log-uniform in [1e-3, 1e2], U a scaled Gaussian, S in [-5, 5]
        u = torch.randn((n, r), generator=g, dtype=torch.float64, device="cuda") / math.sqrt(n)
        a = (u * (10 * torch.rand(r, generator=g, dtype=torch.float64, device="cuda") - 5)) @ u.t()
        s["A"] = 0.5 * (a + a.t())
        s["A"].diagonal().add_(10 ** (5 * torch.rand(n, generator=g, dtype=torch.float64, device="cuda") - 3))
        s["X"] = _block(g, n, c["p"], ld=c["p"])
    elif kind == "syev":
        m = c["s"]
        # a projected matrix V^T AV: Ritz values on the diagonal, couplings to the new directions
        e = 0.05 * torch.randn((m, m), generator=g, dtype=torch.float64, device="cuda")
        s["a"] = 0.5 * (e + e.t())
        s["a"].diagonal().add_(torch.linspace(0.01, 2.0, m, dtype=torch.float64, device="cuda"))
    elif kind == "tridiag":
        n, p = c["n"], c["p"]
        s["d"] = 0.5 + 0.001 * torch.arange(n, device="cuda", dtype=torch.float64) + 0.01 * torch.rand(
            n, generator=g, device="cuda", dtype=torch.float64)
        s["dl"] = 0.02 * torch.randn(n - 1, generator=g, device="cuda", dtype=torch.float64)
        s["du"] = s["dl"].clone()
        s["shift"] = torch.linspace(0.003, 0.02, p, dtype=torch.float64, device="cuda")
        s["R"] = torch.randn((n, p), generator=g, device="cuda", dtype=torch.float64)
    else:
        mixed = c["form"] == "mixed"
        t = _ci(c["n"], seed) if mixed else _cfg1(c["n"], seed)
        more = dict(precision=lb.MIXED, precond=lb.PREC_LEARNED, mlp_weights=lb.load_mlp_weights()) if mixed else {}
        s["solver"] = lb.Solver(**t, extra=c["extra"], **more)
        s["X0"] = _guess(t["diag"], c["k"] + c["extra"])
    return s


# ------------------------------------------------------------------ one pass

def _signed(U):
    """Eigenvectors with their largest entry positive, as a program fixes them that keeps or
    compares them (a sign is arbitrary)."""
    top = U.gather(0, U.abs().argmax(0, keepdim=True))
    return U * torch.where(top < 0, -1.0, 1.0)


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "ortho":
        W = state["W"].copy_(state["W0"])  # both entry points work in place
        return lb.ortho_against(W, state["Y"])[0] if c["q"] else lb.ortho(W)[0]
    if kind == "gram":
        f = dict(f64=lb.gram, df=lb.gram_df, f32=lb.gram_f32_tcgen05)[c["arith"]]
        return f(state["X"], state["Y"])
    if kind == "update":
        f = lb.update_f32 if c["arith"] == "f32" else lb.update_f64_df
        if c["pair"]:
            return f(state["V"], state["U"], AV=state["AV"], lam=state["lam"], resnorm=True)
        return f(state["V"], state["U"])
    if kind == "spmm":
        A = state["A"]
        if c["arith"] == "df":
            return lb.spmm_csr_df(A["row_ptr"], A["col_idx"], A["val"], state["X"], state["Y"])
        return lb.spmm_csr(A["row_ptr"], A["col_idx"], A["val"], state["X"])
    if kind == "dense":
        return lb.spmm_dense(state["A"], state["X"])
    if kind == "syev":
        lam, U = lb.syev(state["a"], two_stage=c["two_stage"])
        return lam, _signed(U)
    if kind == "tridiag":
        return lb.precond_tridiag(state["dl"], state["d"], state["du"], state["shift"], state["R"])
    r = state["solver"].solve(c["k"], c["tol"], X0=state["X0"])
    # a solve to residual tol fixes the vectors to tol / gap: the mixed form's go on in single precision
    return r.evals, r.evecs.float() if c["form"] == "mixed" else r.evecs


# ------------------------------------------------------------------ what it cannot do without

def work(case):
    c = case
    kind = c["kind"]
    if kind == "ortho":
        n, p, q = c["n"], c["p"], c["q"]
        # W read and written, Y read; one projection (two products with Y) and one Cholesky-QR
        return dict(bytes=8 * n * (2 * p + q), flops=n * (4 * p * q + 4 * p * p))
    if kind == "gram":
        b = 4 if c["arith"] == "f32" else 8
        return dict(bytes=b * c["n"] * (c["p"] + c["q"]) + 8 * c["p"] * c["q"], flops=2 * c["n"] * c["p"] * c["q"])
    if kind == "update":
        b, t = (4 if c["arith"] == "f32" else 8), (2 if c["pair"] else 1)
        return dict(bytes=t * b * c["n"] * (3 * c["w"] + c["q"]), flops=t * 2 * c["n"] * 3 * c["w"] * c["q"])
    if kind == "spmm":
        nnz = 65 * c["n"]
        return dict(bytes=12 * nnz + 8 * c["n"] + 16 * c["n"] * c["p"], flops=2 * nnz * c["p"])
    if kind == "dense":
        return dict(bytes=8 * c["n"] ** 2 + 16 * c["n"] * c["p"], flops=2 * c["n"] ** 2 * c["p"])
    if kind == "syev":
        return dict(bytes=16 * c["s"] ** 2, flops=9 * c["s"] ** 3)
    if kind == "tridiag":
        return dict(bytes=24 * c["n"] + 16 * c["n"] * c["p"], flops=12 * c["n"] * c["p"])
    # one iteration at least: the matrix once, the blocks of V and AV once
    n, m = c["n"], c["k"] + c["extra"]
    nnz, b = (65 * n, 4) if c["form"] == "mixed" else (33 * n, 8)
    return dict(bytes=nnz * (b + 4) + 8 * n + 6 * b * n * m, flops=2 * nnz * m + 36 * n * m * m)


# ------------------------------------------------------------------ in 64 bits

def _cholqr(W):
    """The Q of W = Q R with a positive diagonal of R."""
    Q, R = torch.linalg.qr(W)
    return Q * torch.where(R.diagonal() < 0, -1.0, 1.0)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "solve" and (c["form"] == "mixed" or c["n"] > 12_000):
        return None
    s = prepare(case, seed)
    if kind == "ortho":
        W = s["W0"].contiguous()
        if c["q"]:
            for _ in range(2):
                W = W - s["Y"] @ (s["Y"].t() @ W)
        return _cholqr(W)
    if kind == "gram":
        return s["X"].double().t() @ s["Y"].double()
    if kind == "update":
        X = torch.cat([v.double() for v in s["V"]], 1) @ s["U"]
        if not c["pair"]:
            return X
        AX = torch.cat([v.double() for v in s["AV"]], 1) @ s["U"]
        return X, AX, (AX - X * s["lam"]).norm(dim=0)
    if kind == "spmm":
        A, n = s["A"], c["n"]
        return torch.sparse_csr_tensor(A["row_ptr"], A["col_idx"].long(), A["val"], size=(n, n)) @ s["X"].contiguous()
    if kind == "dense":
        return s["A"] @ s["X"]
    if kind == "syev":
        lam, U = torch.linalg.eigh(s["a"])
        return lam, _signed(U)
    if kind == "tridiag":
        # Gaussian elimination down the rows, on the host: T - shift is diagonally dominant here
        d, e, R = s["d"].cpu().numpy(), s["dl"].cpu().numpy(), s["R"].cpu().numpy()
        sh, n = s["shift"].cpu().numpy(), c["n"]
        piv, y = d[0] - sh, R.copy()
        fac = [None] * n
        for i in range(1, n):
            fac[i - 1] = e[i - 1] / piv
            y[i] -= fac[i - 1] * y[i - 1]
            y[i - 1] /= piv
            piv = d[i] - sh - e[i - 1] * fac[i - 1]
        y[n - 1] /= piv
        for i in range(n - 2, -1, -1):
            y[i] -= fac[i] * y[i + 1]
        return torch.from_numpy(y)
    t = _cfg1(c["n"], seed)
    n = c["n"]
    a = torch.sparse_csr_tensor(t["row_ptr"], t["col_idx"].long(), t["val"], size=(n, n)).to_dense()
    lam, U = torch.linalg.eigh(a)
    return lam[:c["k"]], _signed(U[:, :c["k"]])
