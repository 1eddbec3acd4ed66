"""Couplings far below eps ||a|| over normal gaps keep their place in the eigenvectors: a converged pair
of a wide spectrum still has a P direction."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [12, 63, 96])
def test_small_couplings_count(s):
    import torch

    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(s)
    d = np.concatenate([0.003 * np.arange(1, s // 3 + 1), np.sort(rng.uniform(1.0, 2000.0, s - s // 3))])
    a = np.diag(d)
    m = s // 3
    c = 10.0 ** rng.uniform(-13, -9, (m, s - m))  # far below eps ||a|| = 4e-13 many of them
    a[:m, m:], a[m:, :m] = c, c.T
    lam, U = (v.cpu().numpy() for v in lb.syev(torch.from_numpy(a).cuda()))
    assert np.abs(lam - d).max() <= 1e-13 * 2000
    # first order: U[i, j] = a_ij / (d_j - d_i) up to sign, other terms below 1e-12 of it
    U = U * np.sign(np.diagonal(U))
    first = c.T / (d[None, :m] - d[m:, None])
    assert (np.abs(U[m:, :m] - first) <= 1e-6 * np.abs(first)).all()
