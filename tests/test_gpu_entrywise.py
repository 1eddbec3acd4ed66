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
@pytest.mark.parametrize("n,p,q,df", [(40_007, 32, 32, False), (20_000 + 7, 63, 64, False), (9_479, 96, 95, False),
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
