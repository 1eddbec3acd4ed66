"""Dense FP64 product through exact digit products, at the edges of its tiles (64-column panels,
256-row groups, 32-row chunks, row ranges), against extended precision.  Bound: that of the Gram (each
factor held to 2^-56 of the power of two above its column's maximum over 256 rows, left-out products
below 2^-58 * 4 mx my per row, one rounding per group and range)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(1226, 32), (2050, 13), (2560, 5), (4098, 2), (1600, 17), (3001, 7)])
@pytest.mark.parametrize("graded", [False, True])
def test_dense(n, p, graded):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n)
    A, X = rng.standard_normal((n, n)), rng.standard_normal((n, p))
    if graded:
        d = 10.0 ** rng.uniform(-3, 2, n)
        A *= np.sqrt(np.outer(d, d))
        X *= 10.0 ** rng.integers(-20, 20, p)
        X[:300, 0] = 0.0
    A = 0.5 * (A + A.T)
    Y = lb.spmm_dense(torch.from_numpy(A).cuda(), torch.from_numpy(X).cuda()).cpu().numpy()
    ref = A.astype(np.longdouble) @ X.astype(np.longdouble)
    tol = np.zeros((n, p))
    for r in range(0, n, 256):
        a, x = np.abs(A[r:r + 256]), np.abs(X[r:r + 256])
        tol += len(x) * np.outer(a.max(0), x.max(0)) * 2.0**-53
    tol += (n / 256 + 9) * 2.0**-53 * (np.abs(A) @ np.abs(X))
    if n % 2:  # the FMA kernel
        tol = n * 2.0**-53 * (np.abs(A) @ np.abs(X))
    assert (np.abs((Y - ref).astype(np.float64)) <= tol).all()


@pytest.mark.parametrize("n,p", [(1226, 31), (2050, 13)])
def test_both_storage_orders(n, p):
    """Column i of A against X, whichever way A is stored (A is not symmetric here)."""
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n + 1)
    A, X = torch.from_numpy(rng.standard_normal((n, n))).cuda(), torch.from_numpy(rng.standard_normal((n, p))).cuda()
    Y = lb.spmm_dense(A, X)
    assert torch.equal(Y, lb.spmm_dense(A.t().contiguous().t(), X))
    ref = A.t() @ X
    assert (Y - ref).norm() <= 1e-14 * ref.norm()


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200])
@pytest.mark.parametrize("where", ["A", "X"])
def test_outside_the_digits(bad, where):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(1)
    n, p = 2048, 9
    A, X = rng.standard_normal((n, n)), rng.standard_normal((n, p))
    A = 0.5 * (A + A.T)
    if where == "A":
        A[7, 1000] = A[1000, 7] = bad
    else:
        X[1999, 8] = bad
    Y = lb.spmm_dense(torch.from_numpy(A).cuda(), torch.from_numpy(X).cuda()).cpu().numpy()
    with np.errstate(all="ignore"):
        ref = A @ X
        ok = np.isfinite(ref)
        assert (np.isnan(Y) == np.isnan(ref)).all() and (np.isinf(Y) == np.isinf(ref)).all()
        assert (np.abs(Y - ref)[ok] <= (n * 2.0**-52 * (np.abs(A) @ np.abs(X)))[ok]).all()
