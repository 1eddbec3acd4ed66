"""FP64 Gram through exact digit products on the tensor cores, at the edges of its tiles (256-row
groups, 32-row chunks, 32 / 64 / 96 columns), against extended precision.

Bound, per entry and 256-row group g of r rows with column maxima mx, my: both factors are held to
2^-56 of the power of two above the maximum (so 2^-55 mx and 2^-55 my), and the products left out are
below 2^-58 * 4 mx my per row: r mx my (2 * 2^-55 + 2^-56) <= r mx my 2^-53.  One rounding per
group and at most 152 partial sums add (groups + 152) 2^-53 sum |x||y|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _block(x):
    import torch
    n, w = x.shape
    buf = torch.zeros((n, (w + 1) // 2 * 2), dtype=torch.float64, device="cuda")
    buf[:, :w] = torch.from_numpy(x).cuda()
    return buf[:, :w]


def _check(X, Y, C):
    n = X.shape[0]
    ref = X.astype(np.longdouble).T @ Y.astype(np.longdouble)
    tol = np.zeros(ref.shape)
    for r in range(0, n, 256):
        x, y = np.abs(X[r:r + 256]), np.abs(Y[r:r + 256])
        tol += len(x) * np.outer(x.max(0), y.max(0)) * 2.0**-53
    tol += (n / 256 + 153) * 2.0**-53 * (np.abs(X).T @ np.abs(Y))
    err = np.abs((C.astype(np.longdouble) - ref).astype(np.float64))
    assert (err <= tol).all(), (err / np.maximum(tol, 1e-300)).max()


@pytest.mark.parametrize("n,p,q", [(5003, 64, 64), (5120, 63, 65), (5377, 96, 95), (20_011, 32, 33), (40_000, 33, 16),
                                   (65_537, 21, 21), (140_001, 13, 12), (39_171, 42, 21), (330_000, 4, 16)])
@pytest.mark.parametrize("scaled", [False, True])
def test_edges(n, p, q, scaled):
    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n + p)
    X, Y = rng.standard_normal((n, p)), rng.standard_normal((n, q))
    if scaled:  # columns of very different length, localised ones among them, zeros
        X *= 10.0 ** rng.integers(-30, 30, p)
        Y *= 10.0 ** (-12.0 * rng.random((n, q)) ** 4)
        X[:, p // 2] = 0.0
        Y[256:512] = 0.0
    f = lb.gram_df if scaled and n * p * q > 10**8 else lb.gram
    _check(X, Y, _padded(f, X, Y))


def _padded(f, X, Y):
    """Both blocks with one row stride, as the solver lays them out."""
    import torch
    ld = (max(X.shape[1], Y.shape[1]) + 1) // 2 * 2
    out = []
    for v in (X, Y):
        b = torch.zeros((v.shape[0], ld), dtype=torch.float64, device="cuda")
        b[:, :v.shape[1]] = torch.from_numpy(v).cuda()
        out.append(b[:, :v.shape[1]])
    return f(*out).cpu().numpy()


def test_one_block_twice():
    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(5)
    for n, p in ((50_001, 21), (9999, 63)):
        X = rng.standard_normal((n, p))
        b = _block(X)
        _check(X, X, lb.gram(b, b).cpu().numpy())


def test_largest_digits_are_exact():
    """Every row the number whose digits are as negative as they can be: all accumulators at their
    largest, and the sum a whole number that FP64 holds."""
    import paper_2305_06668_gb300 as lb
    n = 8192
    x = -float(0x408080) / 2**23
    X = np.full((n, 64), x)
    C = lb.gram(_block(X), _block(-X)).cpu().numpy()
    assert (C == -n * x * x).all()
    x = -float(0x40808080808080) / 2**55  # all digits but the leading one -128
    X = np.full((n, 64), x)
    _check(X, X, lb.gram(_block(X), _block(X)).cpu().numpy())


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1e200, 5e-324, 1e-200])
def test_outside_the_digits(bad):
    """A block with a number the digits do not hold goes to the FMA kernel."""
    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(9)
    X, Y = rng.standard_normal((6001, 64)), rng.standard_normal((6001, 64))
    X[512:768, 3] = 0.0
    X[600, 3] = bad
    C = lb.gram(_block(X), _block(Y)).cpu().numpy()
    with np.errstate(all="ignore"):
        ref = X.T @ Y
    assert (np.isnan(C) == np.isnan(ref)).all() and (np.isinf(C) == np.isinf(ref)).all()
    ok = np.isfinite(ref)
    bound = 6001 * 2.0**-53 * (np.abs(np.where(np.isfinite(X), X, 0)).T @ np.abs(Y))
    assert (np.abs(C - ref)[ok] <= 2 * bound[ok]).all()
