"""The tensor-core candidate sweep under constant weights, where it jumps between the tiles of
its rows' own tuples: against the f32 candidate sets, on integer components (both exact), over
run layouts and tile counts at which a jump starts, wraps, crosses words of 32 tiles or ends
the sweep.  And the tuple runs of the exact top-k against the full scan on float rows."""
import numpy as np
import pytest

from helpers import dev, empty_out

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CONST = (1.0, 10000.0)


@pytest.fixture(scope="module")
def nhq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_13601_gb300 import build as B

    B.build()
    import paper_2203_13601_gb300 as m

    m.load_library()
    return m


def _runs(layout, N, rng):
    """Run lengths that add up to N."""
    if layout == "even":  # whole tiles and halves of them
        lengths = np.resize([128, 256, 64, 128, 192, 128], 2 + N // 64)
    elif layout == "mixed":  # from below K to several tiles
        lengths = rng.integers(1, 420, N)
    elif layout == "long first":  # one long run, then runs that never fill a list
        lengths = np.r_[N // 2, np.resize([40, 7, 66], N)]
    else:  # long last
        lengths = np.r_[np.resize([90, 130, 70], max(1, N // 200)), N]
    cut = np.minimum(np.cumsum(lengths), N)
    return np.diff(np.r_[0, cut[:np.searchsorted(cut, N) + 1]])


# 1, 31, 32, 33, 64 and 96 tiles, full and cut by one row
@pytest.mark.parametrize("N", [128, 3968, 4095, 4096, 4097, 8192, 12288])
@pytest.mark.parametrize("layout", ["even", "mixed", "long first", "long last"])
@pytest.mark.parametrize("K", [8, 64])
def test_jumping_sweep_finds_the_f32_candidates(nhq, N, layout, K):
    rng = np.random.default_rng(N + K)
    runs = _runs(layout, N, rng)
    tuples = np.repeat(np.arange(runs.size), runs)
    assert tuples.size == N and runs.size < 65536
    order = rng.permutation(N)  # the attribute order has to sort them
    A = np.stack([tuples // 256, tuples % 256], axis=1).astype(np.uint8)[order]
    X = rng.integers(0, 256, (N, 32)).astype(np.float32)
    with nhq.Index.create(dev(X), dev(A), CONST) as ix:
        out = []
        for call in (nhq.nhq_knn, nhq.nhq_knn_bf16):
            ids = torch.empty((N, K), dtype=torch.uint32, device="cuda:0")
            dist = torch.empty((N, K), dtype=torch.float32, device="cuda:0")
            call(ix.handle, K, ids, dist)
            torch.cuda.synchronize()
            out.append((ids.view(torch.int32), dist))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


# both sum a pair's squared differences in dimension order, so every bit agrees
@pytest.mark.parametrize("weights", ["filter", CONST, (1.0, 6.0), (0.5, 0.01)])
@pytest.mark.parametrize("N,nq,d,k", [(50000, 3000, 64, 20), (40000, 60, 100, 5),
                                      (9000, 2500, 32, 33)])
def test_runs_equal_the_scan_on_float_rows(nhq, weights, N, nq, d, k):
    rng = np.random.default_rng(N + nq)
    X = rng.standard_normal((N, d)).astype(np.float32)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    A = rng.integers(0, 3, (N, 2)).astype(np.uint8)
    QA = rng.integers(0, 4, (nq, 2)).astype(np.uint8)  # code 3: no object carries it
    Xd, Qd, pa, pq = dev(X), dev(Q), *(torch.empty(r, dtype=torch.uint32, device="cuda:0")
                                       for r in (N, nq))
    nhq.nhq_pack_attributes(dev(A), pa)
    nhq.nhq_pack_attributes(dev(QA), pq)
    scan, runs = empty_out(nq, k), empty_out(nq, k)
    nhq.nhq_brute_force_noalloc(Xd, pa, 2, Qd, pq, k, *scan, weights=weights)
    with nhq.Index.create(Xd, dev(A), None if weights == "filter" else weights) as ix:
        nhq.nhq_index_build_cells(ix.handle, 4)  # brings the attribute order
        nhq.nhq_brute_force(ix.handle, Qd, dev(QA), k, *runs,
                            weights="filter" if weights == "filter" else "index")
        torch.cuda.synchronize()
    for a, b in zip(scan, runs):
        assert torch.equal(a.view(torch.int32) if a.dtype == torch.uint32 else a,
                           b.view(torch.int32) if b.dtype == torch.uint32 else b)
