"""The exact top-k where its plan and its working memory are at their limits."""
import dataclasses

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


def _check(w, k, ids, g, weights, rows):
    """Rows `rows` of a batch against the oracle, bit for bit (integer components)."""
    got, gam = ids_i64(ids)[rows], g.cpu().numpy()[rows].astype(np.float64)
    if weights == "filter":
        want, wg, _ = O.filtered_topk(w.X, w.A, w.Qv[rows], w.QA[rows], k, prec=O.F32)
    else:
        want, wg, _ = O.fused_topk(w.X, w.A, w.Qv[rows], w.QA[rows], k, weights=weights,
                                   prec=O.F32)
    assert (got == want).all()
    assert np.array_equal(gam[want >= 0], wg[want >= 0])


@pytest.fixture(scope="module")
def warm(nhq):
    """The kernels are loaded (which takes device memory of its own)."""
    w = synth.int_valued(9000, 3000, 32, cards=(2, 3), n_comp=9, seed=1)
    X, A = dev(w.X), dev(w.A)
    with nhq.Index.build(X, A, degree=16, weights=CONST, K=64) as ix:
        for q in (700, 3000):
            for weights in ("filter", "index"):
                ids, g, chi = empty_out(q, 8)
                nhq.nhq_brute_force(ix.handle, dev(w.Qv[:q]), dev(w.QA[:q]), 8, ids, g, chi,
                                    weights=weights)
    torch.cuda.synchronize()


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


# rows of the lists: none (no run reaches two slices), then 89 and 128 MB, beside the plan's
# tables of about 1 MB and, under constant weights, the lists of the queries that are left
# for the scan (at most 20 MB); allocations come in 2 MB pages
@pytest.mark.parametrize("N,nq,k,weights,limit", [
    (1300, 5000, 256, "filter", 8), (60000, 10000, 100, "filter", 96),
    (60000, 10000, 100, CONST, 116), (60000, 10000, 256, CONST, 152)])
def test_working_memory_of_an_exact_batch(nhq, warm, N, nq, k, weights, limit):
    w = synth.int_valued(N, nq, 32, cards=(2, 3), n_comp=9, seed=N)
    with nhq.Index.create(dev(w.X), dev(w.A), CONST) as ix:
        Qv, QA = dev(w.Qv), dev(w.QA)
        ids, g, chi = empty_out(nq, k)
        before = _free()
        nhq.nhq_brute_force(ix.handle, Qv, QA, k, ids, g, chi,
                            weights="filter" if weights == "filter" else "index")
        assert before - _free() <= limit << 20
        _check(w, k, ids, g, weights, np.arange(0, nq, 397))


def test_runs_short_of_list_rows_take_fewer_slices(nhq):
    # k = 256: 65,536 rows; one tuple asks for 4,000 x 45, small ones beside it
    rng = np.random.default_rng(4)
    w = synth.int_valued(100000, 4400, 12, cards=(2, 3, 4), n_comp=9, seed=9)
    often = rng.random(w.N) < 0.9
    w.A, w.QA = w.A.copy(), w.QA.copy()
    w.A[often] = (1, 1, 1)
    w.QA[:4000] = (1, 1, 1)
    for weights in ("filter", CONST):
        with nhq.Index.create(dev(w.X), dev(w.A), CONST) as ix:
            ids, g, chi = empty_out(w.nq, 256)
            nhq.nhq_brute_force(ix.handle, dev(w.Qv), dev(w.QA), 256, ids, g, chi,
                                weights="filter" if weights == "filter" else "index")
            _check(w, 256, ids, g, weights, np.r_[0:4000:211, 4000:4400:31])


def test_an_f32_build_leaves_no_working_memory(nhq, warm):
    w = synth.int_valued(30000, 8, 24, cards=(2, 3), n_comp=9, seed=3)
    X, A = dev(w.X), dev(w.A)
    before = _free()
    with nhq.Index.build(X, A, degree=16, weights=CONST, K=64):
        # rows of 32 floats, two adjacency arrays of 16, the attribute order, reverse lists
        assert before - _free() <= 32 << 20


# the scan and the runs, captured before the index has working memory for them and after,
# then replayed on new queries once larger eager calls have come between
@pytest.mark.parametrize("weights,order", [(None, False), ("filter", True), (CONST, True),
                                           (CONST, False)])
@pytest.mark.parametrize("first", [False, True])
def test_captured_exact_calls_outlive_larger_ones(nhq, warm, weights, order, first):
    w = synth.int_valued(20000, 3000, 48, cards=(2, 3), n_comp=9, seed=13)
    q = 600
    how = "filter" if weights == "filter" else "index"
    with nhq.Index.create(dev(w.X), dev(w.A), weights if weights == CONST else None) as ix:
        if order:
            nhq.nhq_index_build_cells(ix.handle, 4)
        Qv, QA = dev(w.Qv[:q]), dev(w.QA[:q])
        ids, g, chi = empty_out(q, 10)
        if first:
            nhq.nhq_brute_force(ix.handle, Qv[:40], QA[:40], 10, ids[:40], g[:40], chi[:40],
                                weights=how)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            nhq.nhq_brute_force(ix.handle, Qv, QA, 10, ids, g, chi, weights=how)
        big = empty_out(w.nq, 100)
        for other in ("filter", "index"):
            nhq.nhq_brute_force(ix.handle, dev(w.Qv), dev(w.QA), 100, *big, weights=other)
            _check(w, 100, big[0], big[1], "filter" if other == "filter" else
                   (CONST if weights == CONST else None), np.arange(0, w.nq, 501))
        Qv.copy_(dev(w.Qv[q:2 * q]))
        QA.copy_(dev(w.QA[q:2 * q]))
        for _ in range(2):
            ids.zero_()
            g.zero_()
            graph.replay()
            torch.cuda.synchronize()
            part = dataclasses.replace(w, Qv=w.Qv[q:2 * q], QA=w.QA[q:2 * q])
            _check(part, 10, ids, g, weights, np.arange(0, q, 7))
        del graph


def test_attribute_order_of_an_exact_call_serves_other_streams(nhq):
    # the candidate sets make the order on one stream; the search on the other one, which
    # waits for nothing, takes its seeds from it
    w = synth.int_valued(60000, 500, 32, cards=(3, 5), n_comp=9, seed=21)
    X, A, Qv, QA = dev(w.X), dev(w.A), dev(w.Qv), dev(w.QA)
    outs = []
    with nhq.Index.build(X, A, degree=16, weights=CONST, K=32, knn_dtype=1) as built:
        nbr = torch.empty((w.N, 16), dtype=torch.uint32, device="cuda:0")
        nhq.nhq_index_get_graph(built.handle, nbr)
        torch.cuda.synchronize()
    for first in (True, False):
        with nhq.Index.create(X, A, CONST) as ix:
            nhq.nhq_index_set_graph(ix.handle, nbr)
            cand = torch.empty((w.N, 32), dtype=torch.uint32, device="cuda:0")
            ids, g, chi = empty_out(w.nq, 10)
            torch.cuda.synchronize()
            s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
            if first:
                nhq.nhq_knn(ix.handle, 32, cand, stream=s1)
            nhq.nhq_search(ix.handle, Qv, QA, 10, 32, ids, g, chi, seed=1,
                           seed_mode=nhq.SEED_ATTRIBUTE, stream=s2)
            torch.cuda.synchronize()
            outs.append((ids_i64(ids), g.cpu().numpy()))
    assert (outs[0][0] == outs[1][0]).all() and np.array_equal(outs[0][1], outs[1][1])


# runs of all objects, of a half and of a third, in one slice and in several, under weights
# for which none, some or all of the queries are finished by their run: all of them are
# judged after 512 objects
@pytest.mark.parametrize("N,nq,k,cards", [(9000, 300, 10, (1,)), (9000, 300, 256, (2,)),
                                          (24000, 2500, 33, (2,)), (700, 40000, 5, (3,)),
                                          (20000, 2100, 1, (3,))])
@pytest.mark.parametrize("wl", [0.01, 60.0, 120.0, 240.0, 10000.0])
def test_long_runs_under_weak_and_strong_weights(nhq, N, nq, k, cards, wl):
    w = synth.int_valued(N, nq, 32, cards=cards, n_comp=9, seed=N + nq + k)
    with nhq.Index.create(dev(w.X), dev(w.A), (1.0, wl)) as ix:
        nhq.nhq_index_build_cells(ix.handle, 4)  # brings the attribute order
        ids, g, chi = empty_out(nq, k)
        nhq.nhq_brute_force(ix.handle, dev(w.Qv), dev(w.QA), k, ids, g, chi)
        _check(w, k, ids, g, (1.0, wl), np.arange(0, nq, max(1, nq // 300)))
