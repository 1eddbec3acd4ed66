"""The two-stage eigensolver's tolerance: what U^T a U has off the diagonal is at most tol ||a||_F, for every
tol, beside the rounding of s products (s 2^-53 ||a||_F); U is orthonormal to about tol."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tol", [1e-12, 5e-12, 3e-11, 1e-10, 1e-8])
@pytest.mark.parametrize("s", [3, 12, 31, 63, 96])
def test_off_diagonal_mass(s, tol):
    import torch

    import paper_2305_06668_gb300 as lb
    for seed in range(10):
        g = np.random.default_rng(seed)
        e = 10.0 ** g.uniform(-3, 0) * g.standard_normal((s, s))
        a = 0.5 * (e + e.T) + np.diag(np.linspace(0.01, 10.0 ** g.uniform(-2, 2), s))
        _, U = (v.cpu().numpy().astype(np.longdouble) for v in
                lb.syev(torch.from_numpy(a).cuda(), two_stage=True, tol=tol))
        S = U.T @ a.astype(np.longdouble) @ U
        off = float(np.sqrt(((S - np.diag(np.diag(S))) ** 2).sum()))
        nrm = np.linalg.norm(a)
        assert off <= (tol + 4 * s * 2.0**-53) * nrm, (seed, off / nrm)
        assert np.abs((U.T @ U - np.eye(s)).astype(float)).max() <= tol + 4 * (s + 4) * 2.0**-53, seed
