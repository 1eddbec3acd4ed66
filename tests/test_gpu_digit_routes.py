"""Routes to the digit Gram that the tests of its tiles do not take: lobpcg_gram_f64_df above its size rule, one
block behind both operands with more than 64 columns (the diagonal column blocks share their tiles), and
calls from several threads.  Bound as in test_gpu_gram_digits.py."""
import threading

import numpy as np
import pytest

from tests.test_gpu_gram_digits import _block, _check, _padded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,q", [(16_001, 63, 65), (70_003, 32, 31), (9_001, 96, 90), (400_003, 12, 13)])
def test_double_float_entry(n, p, q):
    import paper_2305_06668_gb300 as lb
    rng = np.random.default_rng(n)
    X, Y = rng.standard_normal((n, p)), rng.standard_normal((n, q))
    _check(X, Y, _padded(lb.gram_df, X, Y))


@pytest.mark.parametrize("n,p", [(5_121, 96), (6_007, 95), (12_033, 65)])
def test_wide_block_with_itself(n, p):
    import paper_2305_06668_gb300 as lb
    X = np.random.default_rng(n).standard_normal((n, p))
    b = _block(X)
    _check(X, X, lb.gram(b, b).cpu().numpy())


def test_threads():
    """Each call has its own exponents, flag and error word: whole numbers come out exact on every thread."""
    import torch

    import paper_2305_06668_gb300 as lb
    bad = []

    def work(seed):
        with torch.cuda.stream(torch.cuda.Stream()):
            g = torch.Generator(device="cuda")
            g.manual_seed(seed)
            for n, p in ((60_001, 21), (9_001, 64), (11_003, 96)):
                X = torch.randint(-8, 9, (n, p + p % 2), generator=g, device="cuda").double()[:, :p]
                ref = X.t() @ X
                for _ in range(6):
                    if not torch.equal((lb.gram_df if seed & 1 else lb.gram)(X, X), ref):
                        bad.append((seed, n, p))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad
