"""df_products = -1: FP64 fused multiply-adds in every FP64 product, also at the sizes from which the other
settings take digit products on the tensor cores."""
import numpy as np
import pytest

import synth
from tests.gpu_util import cuda, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", [False, True])
def test_minus_one_is_another_arithmetic(dense):
    """Above the size rules the two settings round differently; both reach the same pairs."""
    torch = cuda()
    import paper_2305_06668_gb300 as lb
    if dense:  # the product with A is the only one above its rule
        n, k = 2048, 4
        diag = 0.01 * np.arange(1, n + 1)
        A = 1e-3 * np.random.default_rng(11).standard_normal((n, n))
        A = 0.5 * (A + A.T)
        np.fill_diagonal(A, diag)
        mat = dict(dense=dev(torch, A), diag=dev(torch, diag))
    else:
        n, k = 100_003, 8
        a = synth.sparse_cfg1(n=n, seed=11)
        mat, diag = lb.upload_csr(a), a.diag
    x0 = dev(torch, synth.diag_guess(diag, k + 4, seed=11))
    out = {}
    for df in (0, -1):
        s = lb.Solver(**mat, extra=4, df_products=df)
        out[df] = s.solve(k, 1e-9, X0=x0)
        s.close()
        assert out[df].status == lb.OK
    assert np.abs(out[0].evals - out[-1].evals).max() <= 1e-12 * max(1.0, np.abs(out[0].evals).max())
    assert not torch.equal(out[0].evecs, out[-1].evecs)


def test_profile_tells_the_digit_updates():
    torch = cuda()
    import paper_2305_06668_gb300 as lb
    n, k = 100_003, 8
    a = synth.sparse_cfg1(n=n, seed=11)
    x0 = dev(torch, synth.diag_guess(a.diag, k + 4, seed=11))
    for df in (0, -1):
        s = lb.Solver(**lb.upload_csr(a), extra=4, df_products=df, profile=True)
        i = s.solve(k, 1e-9, X0=x0).info
        s.close()
        assert 0 <= i["update_digit_launches"] <= i["update_fp64_launches"]
        assert (i["update_digit_launches"] > 0) == (df == 0)
        assert (i["update_digit_flops"] > 0) == (i["update_digit_seconds"] > 0) == (df == 0)
        assert i["update_digit_seconds"] <= i["update_fp64_seconds"]
