"""The cluster eigensolver (FP32 Jacobi, FP64 refinement) at sizes around its split over eight CTAs, on
spectra that FP32 does not separate: eigenvalues and residuals to 1e-13 ||a||, U orthonormal to
1e-13 s (the bounds that the plain Jacobi solver is held to)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(kind, s, g):
    Q = np.linalg.qr(g.standard_normal((s, s)))[0]
    lam = np.sort(g.uniform(-1, 1, s))
    if kind == "pairs":      # a 2 x 2 block structure with equal diagonals: angles of 45 degrees
        a = np.diag(np.repeat(np.arange((s + 1) // 2), 2)[:s].astype(float))
        for i in range(0, s - 1, 2):
            a[i, i + 1] = a[i + 1, i] = 1e-9
        return a
    if kind == "close":      # gaps down to 1e-10
        lam[s // 2:] = lam[s // 2] + np.cumsum(10.0 ** g.uniform(-10, -6, s - s // 2))
    if kind == "repeated":
        lam[: s // 2 + 1] = 0.25
    if kind == "graded":     # Ritz values on the diagonal, small couplings, wide range
        a = 1e-3 * g.standard_normal((s, s)) * np.sqrt(np.outer(*[10.0 ** np.linspace(-3, 2, s)] * 2))
        return 0.5 * (a + a.T) + np.diag(10.0 ** np.linspace(-3, 2, s))
    if kind == "diagonal":
        return np.diag(lam)
    if kind == "scaled":
        lam = lam * 1e150
    if kind == "zero":
        lam = 0 * lam
    a = (Q * lam) @ Q.T
    return 0.5 * (a + a.T)


@pytest.mark.parametrize("two_stage", [False, True])
@pytest.mark.parametrize("kind", ["plain", "pairs", "close", "repeated", "graded", "diagonal", "scaled", "zero"])
@pytest.mark.parametrize("s", [2, 3, 8, 9, 17, 63, 64, 96])
def test_spectra(s, kind, two_stage):
    import torch

    import paper_2305_06668_gb300 as lb
    a = _matrix(kind, s, np.random.default_rng(s))
    lam, U = (v.cpu().numpy() for v in lb.syev(torch.from_numpy(a).cuda(), two_stage=two_stage))
    ref = np.linalg.eigvalsh(a)
    nrm = np.linalg.norm(a)
    assert (np.diff(lam) >= 0).all()
    assert np.abs(lam - ref).max() <= 1e-13 * nrm
    assert np.abs(U.T @ U - np.eye(s)).max() <= 1e-13 * s
    assert np.abs(a @ U - U * lam).max() <= 1e-13 * nrm


def test_nan_stays_nan():
    import torch

    import paper_2305_06668_gb300 as lb
    a = np.eye(12)
    a[3, 4] = a[4, 3] = np.nan
    lam, _ = lb.syev(torch.from_numpy(a).cuda())
    assert np.isnan(lam.cpu().numpy()).any()
