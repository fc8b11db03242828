"""The two ways of the exact top-k (tuple runs and full scan) and the tiled gradient of the
entry model, at the edges of their tiles, slices and plans, against the oracle.  Components
are integers, so ids, chi and Gamma are compared bit for bit."""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import dev, empty_out, ids_i64
from oracle import mlp

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


def _check(nhq, w, k, weights, wt, ix):
    ids, g, chi = empty_out(w.nq, k)
    nhq.nhq_brute_force(ix.handle, dev(w.Qv), dev(w.QA), k, ids, g, chi, weights=weights)
    torch.cuda.synchronize()
    got = ids_i64(ids)
    if wt == "filter":
        want, dl, _ = O.filtered_topk(w.X, w.A, w.Qv, w.QA, k, prec=O.F32)
        assert (got == want).all()
        gg = g.cpu().numpy().astype(np.float64)
        assert np.array_equal(gg[want >= 0], dl[want >= 0])
        assert np.isinf(gg[want < 0]).all()
        assert (chi.cpu().numpy()[want < 0] == 255).all()
    else:
        want, wg, wc = O.fused_topk(w.X, w.A, w.Qv, w.QA, k, weights=wt, prec=O.F32)
        assert (got == want).all()
        assert np.array_equal(g.cpu().numpy().astype(np.float64), wg)
        assert (chi.cpu().numpy().astype(np.int64) == wc).all()


# nq 64 | 65: tiles of 4 or 32 queries; 2,048 | 2,049: the plan in one block or in three
# kernels; k above the rarest runs leaves queries to the full scan; d odd: unaligned queries
@pytest.mark.parametrize("N,nq,d,k,cards", [
    (70000, 16, 64, 10, (2, 3)), (30001, 64, 37, 1, (2, 2, 2)), (16000, 65, 68, 33, (3, 5, 7)),
    (2100, 2048, 20, 100, (3, 10, 20)), (1300, 2049, 31, 7, (3, 4)), (129, 5000, 128, 40, (2,)),
])
@pytest.mark.parametrize("weights", ["filter", CONST, (1.0, 30.0)])
def test_tuple_runs_match_the_oracle(nhq, N, nq, d, k, cards, weights):
    w = synth.int_valued(N, nq, d, cards=cards, n_comp=12, seed=N + nq)
    w.QA = w.QA.copy()
    w.QA[::17, 0] = 200  # a code that no object carries: an empty run
    with nhq.Index.create(dev(w.X), dev(w.A), None if weights == "filter" else weights) as ix:
        nhq.nhq_index_build_cells(ix.handle, 4)  # brings the attribute order
        _check(nhq, w, k, "filter" if weights == "filter" else "index", weights, ix)


# tiles of 4, 32 and 64 queries, one and several slices, without the attribute order
@pytest.mark.parametrize("N,nq,d,k", [(1, 3, 5, 1), (127, 8, 33, 128), (5000, 9, 16, 256),
                                      (9000, 1025, 30, 64), (4097, 1500, 64, 100),
                                      (40000, 4, 100, 20)])
@pytest.mark.parametrize("weights", [None, "filter", CONST])
def test_full_scan_matches_the_oracle(nhq, N, nq, d, k, weights):
    w = synth.int_valued(N, nq, d, cards=(2, 3, 4), n_comp=min(N, 12), seed=N + 3 * nq)
    k = min(k, N)
    with nhq.Index.create(dev(w.X), dev(w.A), weights if weights == CONST else None) as ix:
        _check(nhq, w, k, "filter" if weights == "filter" else "index", weights, ix)


def test_scan_of_unaligned_queries_and_runs_of_candidates(nhq):
    # queries that start 4 bytes past a 16-byte boundary, and nhq_knn over the runs
    w = synth.int_valued(6000, 40, 48, cards=(2, 3), n_comp=9, seed=5)
    buf = torch.empty(w.nq * 48 + 1, dtype=torch.float32, device="cuda:0")
    q = buf[1:].view(w.nq, 48)
    q.copy_(dev(w.Qv))
    ids, g, chi = empty_out(w.nq, 12)
    with nhq.Index.create(dev(w.X), dev(w.A), CONST) as ix:
        nhq.nhq_brute_force(ix.handle, q, dev(w.QA), 12, ids, g, chi)
        cand = torch.empty((w.N, 16), dtype=torch.uint32, device="cuda:0")
        dist = torch.empty((w.N, 16), dtype=torch.float32, device="cuda:0")
        nhq.nhq_knn(ix.handle, 16, cand, dist)
    torch.cuda.synchronize()
    want, wg, _ = O.fused_topk(w.X, w.A, w.Qv, w.QA, 12, weights=CONST, prec=O.F32)
    assert (ids_i64(ids) == want).all()
    assert np.array_equal(g.cpu().numpy().astype(np.float64), wg)
    pick = np.arange(0, w.N, 61)
    self_ids, self_g, _ = O.fused_topk(w.X, w.A, w.X[pick], w.A[pick], 17, weights=CONST,
                                       prec=O.F32)
    got, gd = ids_i64(cand)[pick], dist.cpu().numpy().astype(np.float64)[pick]
    for row, u in enumerate(pick):
        keep = self_ids[row] != u
        assert (got[row] == self_ids[row][keep][:16]).all()
        assert np.array_equal(gd[row], self_g[row][keep][:16])


@pytest.mark.parametrize("d,E,n", [(1, 1, 1), (63, 65, 127), (64, 64, 129), (65, 130, 300),
                                   (200, 63, 1025)])
def test_entry_gradient_at_the_edges_of_its_tiles(nhq, d, E, n):
    rng = np.random.default_rng(d * E + n)
    p = (rng.standard_normal(mlp.entry_size(d, E)) * 0.2).astype(np.float32)
    p[0] = 0.5 / np.sqrt(d)
    Q = rng.standard_normal((n, d)).astype(np.float32)
    y = rng.integers(0, E, n).astype(np.int32)
    if n > 1:
        y[::31] = E  # ignored samples
    grad = torch.empty(p.size, dtype=torch.float32, device="cuda:0")
    loss = torch.empty(1, dtype=torch.float32, device="cuda:0")
    nhq.nhq_entry_grad(dev(p), E, dev(Q), dev(y), grad, loss)
    torch.cuda.synchronize()
    keep = y < E
    lw, gw = mlp.entry_loss_and_grad(p.astype(np.float64), Q[keep], y[keep], d, E)
    frac = keep.sum() / n
    # f32 sums of at most 1,025 terms: relative 1e-4 of each sum's largest terms
    assert abs(loss.item() - lw * frac) <= 1e-4 * max(abs(lw), 1e-3)
    assert np.allclose(grad.cpu().numpy(), gw * frac, rtol=1e-3, atol=1e-5 * np.abs(gw).max())


def test_exact_queries_leave_a_captured_search_alone(nhq):
    # the exact calls' working memory is larger than the search's, whose address the
    # captured search keeps
    w = synth.int_valued(20000, 3000, 16, cards=(2, 3), n_comp=9, seed=8)
    q = 50
    with nhq.Index.build(dev(w.X), dev(w.A), degree=16, weights=CONST, K=32) as ix:
        ids, g, chi = empty_out(q, 10)
        Qv, QA = dev(w.Qv[:q]), dev(w.QA[:q])  # the captured search reads them at every launch
        graph = nhq.nhq_search_graph_create(ix.handle, Qv, QA, 10, 32, ids, g, chi, seed=1,
                                            seed_mode=nhq.SEED_ATTRIBUTE)
        torch.cuda.synchronize()
        want = ids_i64(ids), g.cpu().numpy().copy()
        for weights in ("filter", "index", None):
            _check(nhq, w, 10, weights, CONST if weights == "index" else weights, ix)
        ids.zero_()
        g.zero_()
        graph.launch()
        torch.cuda.synchronize()
        assert (ids_i64(ids) == want[0]).all() and np.array_equal(g.cpu().numpy(), want[1])
        graph.close()
