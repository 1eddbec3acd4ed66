"""U of the eigensolvers is orthonormal to FP64 rounding also where eigenvalues are so close that rounding
turns the vectors: many gaps of 1e-10 ||a||.  A last step X + X E with |E| <= 1e-9 rounds an entry once, and
E holds the rounding of inner products of s terms: |U^T U - I| <= (s + 4) 2^-53, and four times that is asked
for.  (Larger s with this many close gaps take the Jacobi rotations behind the refinement, whose rounding
grows with (s - 1) sweeps rotations a column; tests/test_gpu_syev_cluster.py holds them.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("two_stage", [False, True])
@pytest.mark.parametrize("s", [5, 8, 10, 12, 16, 24])
def test_small_gaps(s, two_stage):
    import torch

    import paper_2305_06668_gb300 as lb
    for seed in range(12):
        g = np.random.default_rng(seed)
        Q = np.linalg.qr(g.standard_normal((s, s)))[0]
        lam = np.sort(g.uniform(-1, 1, s))
        lam[s // 2:] = lam[s // 2] + np.cumsum(10.0 ** g.uniform(-10.5, -9, s - s // 2))
        a = (Q * lam) @ Q.T
        a = 0.5 * (a + a.T)
        ev, U = (v.cpu().numpy() for v in lb.syev(torch.from_numpy(a).cuda(), two_stage=two_stage))
        Ul = U.astype(np.longdouble)
        assert np.abs((Ul.T @ Ul - np.eye(s)).astype(float)).max() <= 4 * (s + 4) * 2.0**-53, seed
        assert np.abs(a @ U - U * ev).max() <= 1e-13 * np.linalg.norm(a)
