"""The FP64 building blocks on columns and rows whose entries are far apart.  Above their size rules they run
on digits that share one power of two per column and 256 rows (Gram, dense product) or per row (update); what
such a digit drops may be all there is in another entry.  These inputs are held to the bounds of the
arithmetic without digits, entry by entry: n 2^-53 |X|^T|Y| for a chain of fused multiply-adds, and
(8 + k) 2^-47 |X|^T|Y| for double-float sums of k terms between two FP64 adds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FMA, DF = 2.0**-53, 2.0**-47


def _one_stride(*blocks):
    import torch
    ld = (max(b.shape[1] for b in blocks) + 1) // 2 * 2
    out = []
    for v in blocks:
        b = torch.zeros((v.shape[0], ld), dtype=torch.float64, device="cuda")
        b[:, :v.shape[1]] = torch.from_numpy(v).cuda()
        out.append(b[:, :v.shape[1]])
    return out


def _far_apart(kind, n, p, q, rng):
    X, Y = rng.standard_normal((n, p)), rng.standard_normal((n, q))
    if kind == "spikes":  # one entry of X per 256 rows stands out, where Y vanishes
        X *= 1e-9
        X[5::256], Y[5::256] = 1.5, 0.0
    elif kind == "alternate":  # large where the other is small
        X[::2] *= 1e-18
        Y[1::2] *= 1e-18
    elif kind == "tail":  # only the last rows, fewer than 256, and only one of them counts in X
        X[:-7] = 0.0
        X[-7:] *= 1e-12
        X[-3], Y[-3] = 1.0, 0.0
    elif kind == "one pair":  # a single pair of columns
        X[:, p - 1] *= 1e-9
        X[300, p - 1], Y[300, 0] = 1.5, 0.0
        X[301:512, p - 1] = 0.0
    return X, Y


@pytest.mark.parametrize("kind", ["spikes", "alternate", "tail", "one pair"])
@pytest.mark.parametrize("n,p,q,df", [(20_007, 32, 32, False), (9_607, 63, 64, False), (9_479, 96, 95, False),
                                      (70_007, 33, 32, True)])
def test_gram(n, p, q, df, kind):
    import paper_2305_06668_gb300 as lb
    X, Y = _far_apart(kind, n, p, q, np.random.default_rng(n))
    got = (lb.gram_df if df else lb.gram)(*_one_stride(X, Y)).cpu().numpy()
    ref = X.astype(np.longdouble).T @ Y.astype(np.longdouble)
    size = np.abs(X).T @ np.abs(Y)
    tol = (136 * DF if df else n * FMA) * size
    err = np.abs((got.astype(np.longdouble) - ref).astype(np.float64))
    assert (err <= tol).all(), (err / np.maximum(tol, 1e-300)).max()


def _rows_far_apart(kind, n, s, q, rng):
    V, U = rng.standard_normal((n, s)), np.zeros((s, q))
    if kind == "lengths":  # columns of V of different length, each an output of its own
        V *= 10.0 ** -np.linspace(0, 12, s)
        U[:q, :q] = np.eye(q)
    elif kind == "pairs of rows":  # a few rows only, two outputs
        V[::97, 0], V[::97, 1] = 1e10, 1e-10
        U[:q, :q] = np.eye(q)
        U += 1e-30 * rng.standard_normal((s, q))
    elif kind == "last row":
        V[n - 1, 2:] = 0.0
        V[n - 1, :2] = 1.0, 1e-13
        U[:] = rng.standard_normal((s, q))
        U[0, 1:] = 0.0
    elif kind == "column of U":  # an output that only the row's smallest entries reach
        U[:] = rng.standard_normal((s, q))
        U[:s - 1, q - 1] = 0.0
        V[:, s - 1] *= 1e-12
    return V, U


@pytest.mark.parametrize("kind", ["lengths", "pairs of rows", "last row", "column of U"])
@pytest.mark.parametrize("n,s,q,pair", [(46_001, 63, 21, False), (15_011, 64, 32, True), (73_003, 32, 13, True),
                                        (20_003, 96, 32, False)])
@pytest.mark.parametrize("in_place", [False, True])
def test_update(n, s, q, pair, in_place, kind):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n)
    V, U = _rows_far_apart(kind, n, s, q, rng)
    W = rng.standard_normal((n, s)) * np.abs(V)
    (Vt,), (Wt,) = _one_stride(V), _one_stride(W)
    more = dict(AV=[Wt], lam=torch.zeros(q, dtype=torch.float64, device="cuda"), resnorm=True) if pair else {}
    if in_place:
        more.update(dict(X=Vt, AX=Wt) if pair else dict(X=Vt))
    got = lb.update_f64_df([Vt], torch.from_numpy(U).cuda(), alpha=-1.0, **more)
    for o, x in zip(got[:2] if pair else [got], [V, W]):
        ref = -(x.astype(np.longdouble) @ U.astype(np.longdouble))
        tol = (s + 8) * DF * (np.abs(x) @ np.abs(U))
        err = np.abs((o.cpu().numpy()[:, :q].astype(np.longdouble) - ref).astype(np.float64))
        assert (err <= tol).all(), (err / np.maximum(tol, 1e-300)).max()


@pytest.mark.parametrize("kind", ["spikes", "alternate", "tail", "diagonal"])
@pytest.mark.parametrize("n,p", [(2048, 5), (2050, 13), (1226, 32)])
def test_dense(n, p, kind):
    """Column i of A against X; the FMA kernel where an entry asks for it, in either storage order."""
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n + p)
    if kind == "diagonal":  # dominant, and X without the rows it would meet
        A, X = 1e-3 * rng.standard_normal((n, n)), rng.standard_normal((n, p))
        np.fill_diagonal(A, 1e8)
        X[::64] = 0.0
    else:
        A, X = _far_apart(kind, n, n, p, rng)
    ref = A.T.astype(np.longdouble) @ X.astype(np.longdouble)
    tol = n * FMA * (np.abs(A).T @ np.abs(X))
    At, Xt = torch.from_numpy(A).cuda(), torch.from_numpy(X).cuda()
    for a in (At, At.t().contiguous().t()):
        err = np.abs((lb.spmm_dense(a, Xt).cpu().numpy().astype(np.longdouble) - ref).astype(np.float64))
        assert (err <= tol).all(), (err / np.maximum(tol, 1e-300)).max()
