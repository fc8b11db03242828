"""The exact top-k where its plan and its working memory are at their limits."""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import dev, empty_out, ids_i64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CONST = (1.0, 10000.0)


@pytest.fixture(scope="module")
def nhq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_13601_gb300 import build as B

    B.build()
    O.build()
    import paper_2203_13601_gb300 as m

    m.load_library()
    return m


def test_more_than_2_24_tuples_in_one_batch(nhq):
    # every object has a tuple of its own and every query asks for one of them
    n = (1 << 24) + 1000
    i = torch.arange(n, device="cuda:0")
    A = torch.stack([(i >> s) & 255 for s in (0, 8, 16, 24)], dim=1).to(torch.uint8)
    g = torch.Generator(device="cuda:0")
    g.manual_seed(7)
    X = torch.randint(0, 256, (n, 4), generator=g, device="cuda:0").to(torch.float32)
    pick = torch.randperm(n, generator=g, device="cuda:0")
    ids, dist, chi = empty_out(n, 1)
    with nhq.Index.create(X, A, None) as ix:
        nhq.nhq_brute_force(ix.handle, X[pick], A[pick].contiguous(), 1, ids, dist, chi,
                            weights="filter")
        torch.cuda.synchronize()
    assert torch.equal(ids.view(torch.int32)[:, 0].long(), pick)
    assert not dist.any() and not chi.any()
