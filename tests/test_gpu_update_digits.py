"""FP64 block updates through exact digit products on the tensor cores, at the edges of their tiles
(128-row tiles, 8-row copies, 32-column chunks, 4-column groups), against extended precision.

Bound, entry (i, j): with g_l the largest |alpha U_lj| of row l, R_i = max_l 2 |V_il| g_l bounds the
scaled row and C_j = max_l |alpha U_lj| / g_l the scaled column; both factors are held to 2^-56 of the
power of two above, and the products left out are below 2^-58 * 4 R C each: s R_i C_j 2^-53.  The
rounding of alpha U, of the sum and of the base's add add 2^-52 (sum |V||U| + |base|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _blocks(v, ws, ld):
    import torch
    out, o = [], 0
    for w in ws:
        b = torch.zeros((v.shape[0], ld), dtype=torch.float64, device="cuda")
        b[:, :w] = torch.from_numpy(v[:, o:o + w].copy()).cuda()
        out.append(b[:, :w])
        o += w
    return out


def _reference(V, U, alpha, base=None):
    A = alpha * U
    ref = V.astype(np.longdouble) @ A.astype(np.longdouble)
    aV, aA = np.abs(V), np.abs(A)
    g = np.maximum(aA.max(1), 1e-300)
    R, C = 2 * (aV * g).max(1), (aA / g[:, None]).max(0)
    tol = V.shape[1] * np.outer(R, C) * 2.0**-53 + 2.0**-52 * (aV @ aA)
    if base is not None:
        ref = ref + base
        tol = tol + 2.0**-52 * np.abs(base)
    return ref, tol


def _ok(got, ref, tol):
    err = np.abs((got.cpu().numpy().astype(np.longdouble) - ref).astype(np.float64))
    assert (err <= tol).all(), (err / np.maximum(tol, 1e-300)).max()


@pytest.mark.parametrize("n,ws,q", [(50_003, (21, 21, 21), 21), (128 * 310 + 1, (32, 32, 32), 32), (130_001, (21,), 23),
                                    (200_001, (17, 2, 15), 9), (40_007, (64,), 32), (60_009, (33, 31), 17),
                                    (1_100_001, (8, 4, 5), 4)])
@pytest.mark.parametrize("graded", [False, True])
def test_update(n, ws, q, graded):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n)
    s, ld = sum(ws), (max(ws) + 1) // 2 * 2
    V, U = rng.standard_normal((n, s)), np.linalg.qr(rng.standard_normal((96, 96)))[0][:s, :q].copy()
    if graded:  # columns of V of very different length met by rows of U, sparse rows, a zero row of U
        f = 10.0 ** rng.integers(-20, 20, s)
        V, U = V * f, U / f[:, None] * 10.0 ** rng.integers(-3, 3, q)
        V *= 10.0 ** (-10 * rng.random((n, 1)))
        V[::7] = 0.0
        U[s // 2] = 0.0
    base = rng.standard_normal((n, q))
    Vt, Ut, bt = _blocks(V, ws, ld), torch.from_numpy(U).cuda(), torch.from_numpy(base).cuda()
    ref, tol = _reference(V, U, -1.0, base)
    _ok(lb.update_f64_df(Vt, Ut, alpha=-1.0, base=bt), ref, tol)
    _ok(lb.update_f64_df(Vt, Ut, alpha=-1.0, base=bt, X=bt), ref, tol)  # in place on the base


@pytest.mark.parametrize("n,ws,q", [(40_001, (21, 21, 21), 21), (20_130, (32, 32, 32), 31), (200_003, (13,), 13)])
def test_pair_with_norms(n, ws, q):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n + 1)
    s, ld = sum(ws), (max(ws) + 1) // 2 * 2
    V, W, U = rng.standard_normal((n, s)), rng.standard_normal((n, s)), rng.standard_normal((s, q))
    lam = rng.standard_normal(q)
    X, AX, rn = lb.update_f64_df(_blocks(V, ws, ld), torch.from_numpy(U).cuda(), AV=_blocks(W, ws, ld),
                                 lam=torch.from_numpy(lam).cuda(), resnorm=True)
    for got, v in ((X, V), (AX, W)):
        _ok(got, *_reference(v, U, 1.0))
    r = AX.cpu().numpy() - X.cpu().numpy() * lam
    assert np.allclose(rn, np.linalg.norm(r, axis=0), rtol=1e-13, atol=0)


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200, 1e-200, 5e-324])
@pytest.mark.parametrize("where", ["V", "U"])
def test_outside_the_digits(bad, where):
    """Rows (or a U) that the digits do not hold are formed with FP64 FMAs, in place too."""
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(3)
    n, s = 100_001, 32
    V, U = rng.standard_normal((n, s)), rng.standard_normal((s, s))
    if where == "V":
        V[5000], V[n - 1], V[77, 3] = 0.0, 0.0, bad
        V[5000, 7] = V[n - 1, 31] = bad
    else:
        U[:, 4] = 0.0
        U[9, 4] = bad
    Vt, Ut = _blocks(V, (s,), s), torch.from_numpy(U).cuda()
    got = lb.update_f64_df(Vt, Ut, X=Vt[0]).cpu().numpy()
    with np.errstate(all="ignore"):
        ref = V @ U
        tol = 64 * 2.0**-52 * (np.abs(V) @ np.abs(U)) + 1e-320
    assert (np.isnan(got) == np.isnan(ref)).all() and (np.isinf(got) == np.isinf(ref)).all()
    ok = np.isfinite(ref)
    if where == "V":
        assert (np.abs(got - ref)[ok] <= tol[ok]).all()
    else:
        m = np.delete(np.arange(s), 4)
        f = ok[:, m]
        assert (np.abs(got - ref)[:, m][f] <= tol[:, m][f]).all()
        if np.isfinite(bad):
            assert (np.abs(got - ref)[:, 4] <= tol[:, 4]).all()
