"""The eigensolvers with U in a's own memory, on a spectrum that takes the refinement's scratch writes to U and
then the Jacobi kernel behind it (half of the eigenvalues within 1e-8 ||a|| of each other)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("two_stage", [False, True])
@pytest.mark.parametrize("s", [17, 63, 96])
def test_vectors_over_the_matrix(s, two_stage):
    import torch

    import paper_2305_06668_gb300 as lb
    g = np.random.default_rng(s)
    Q = np.linalg.qr(g.standard_normal((s, s)))[0]
    ev = np.sort(g.uniform(-1, 1, s))
    ev[s // 2:] = ev[s // 2] + np.cumsum(10.0 ** g.uniform(-10.5, -9, s - s // 2))
    a = (Q * ev) @ Q.T
    a = 0.5 * (a + a.T)
    buf, lam = torch.from_numpy(a).cuda(), torch.empty(s, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p, l = ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(lam.data_ptr())
    L = lb.lib()
    st = (L.lobpcg_syev2_f64(ctypes.c_int(s), p, ctypes.c_double(0.0), l, p, None) if two_stage
          else L.lobpcg_syev_f64(ctypes.c_int(s), p, l, p, None))
    assert st == lb.OK
    U, lam = buf.cpu().numpy().T, lam.cpu().numpy()  # column-major
    assert np.abs(lam - ev).max() <= 1e-13 * np.linalg.norm(a)
    assert np.abs(U.T @ U - np.eye(s)).max() <= 1e-13 * s
    assert np.abs(a @ U - U * lam).max() <= 1e-13 * np.linalg.norm(a)


@pytest.mark.parametrize("tol", [0.0, 1e-10])
@pytest.mark.parametrize("s", [2, 3, 9, 63, 96])
def test_two_stage_kernel_by_itself(s, tol):
    """U over the matrix always takes the two-stage Jacobi kernel: both of its polishing forms."""
    import torch

    import paper_2305_06668_gb300 as lb
    g = np.random.default_rng(s)
    e = 0.05 * g.standard_normal((s, s))
    a = 0.5 * (e + e.T) + np.diag(np.linspace(0.01, 2.0, s))
    buf, lam = torch.from_numpy(a).cuda(), torch.empty(s, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p, l = ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(lam.data_ptr())
    assert lb.lib().lobpcg_syev2_f64(ctypes.c_int(s), p, ctypes.c_double(tol), l, p, None) == lb.OK
    U, lam, nrm = buf.cpu().numpy().T, lam.cpu().numpy(), np.linalg.norm(a)
    assert (np.diff(lam) >= 0).all()
    assert np.abs(lam - np.linalg.eigvalsh(a)).max() <= (1e-13 + tol) * nrm
    assert np.abs(U.T @ U - np.eye(s)).max() <= 1e-13 * s + tol
    assert np.abs(a @ U - U * lam).max() <= (1e-13 + tol) * nrm
