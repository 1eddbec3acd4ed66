"""The workspace pool of the building-block entry points: calls from several threads on their own
streams get their own memory, and trimming gives it back without touching later calls."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_threads_and_trim():
    import torch

    import paper_2305_06668_gb300 as lb

    bad = []

    def work(seed):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            g = torch.Generator(device="cuda")
            g.manual_seed(seed)
            for n, p in ((4096, 4), (20_001, 21), (777, 6)):
                X = torch.randint(-8, 9, (n, p + p % 2), generator=g, device="cuda").double()[:, :p]
                for _ in range(5):
                    C = lb.gram(X, X)
                    if not torch.equal(C, X.t() @ X):  # whole numbers: exact in any order
                        bad.append((seed, n, p))
                if seed == 0:
                    lb.trim_workspace()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    lb.trim_workspace()
    assert not bad
