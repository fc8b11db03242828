"""Workloads whose speed counts: hybrid-query search, exact search and index construction
as a program calls them through ``paper_2203_13601_gb300``.

A case is a dict of plain values.  ``kind`` picks the call:

* ``search``   ``nhq_search`` on a built graph (one k and ef for the batch)
* ``batched``  ``nhq_search_batched``, every query with its own k and ef
* ``brute``    ``nhq_brute_force``, the exact answer over all objects
* ``knn``      ``nhq_knn``, the exact candidate sets of the f32 build
* ``build``    ``Index.build`` with tensor-core candidates: raw vectors to finished graph
* ``entry``    ``nhq_entry_grad``, one forward and backward pass of the entry model

Objects and queries are drawn from one mixture of clusters (the shape of the paper's
sets): ``data`` "int" has integer components 0..255, "float" is Gaussian, "unit" is
Gaussian with unit rows.  Attributes are ordinal codes with the cardinalities of
``cards``, uniform or Zipf (s = 1).  ``weights``: "constant" is (w_v, w_l) = (1, 10000),
where a matching tuple outranks any distance; "proportional" is the default weighting of
the fusion distance; "filter" asks for exact matches only (the ground truth of hybrid
recall).
"""
import math

import torch

import paper_2203_13601_gb300 as nhq

DEVICE = "cuda:0"
DEGREE, CANDIDATES = 32, 64
VEC = {"f32": nhq.VEC_F32, "bf16": nhq.VEC_BF16, "f16": nhq.VEC_F16, "fp8": nhq.VEC_FP8E4M3}
SEEDS = {"random": nhq.SEED_RANDOM, "attribute": nhq.SEED_ATTRIBUTE,
         "nearest": nhq.SEED_ATTRIBUTE_NEAR}


def _search(name, n, d, q, k, ef, **kw):
    c = dict(name=name, kind="search", n=n, d=d, q=q, k=k, ef=ef, data="int", comps=1000,
             cards="3/10/20", zipf=True, weights="constant", vec="f32", rerank=False,
             seeds="attribute")
    c.update(kw)
    return c


def listed():
    return [
        # one interactive query on a small collection: launches and the dependent chain count
        _search("search_one", 10_000, 128, 1, 10, 64, data="float", comps=100, cards="3/5/10",
                zipf=False),
        # a batch on a small collection with every option at its default (random entry
        # points, proportional weighting)
        _search("search_small", 10_000, 128, 1_000, 10, 100, data="float", comps=100,
                cards="3/5/10", zipf=False, weights="proportional", seeds="random"),
        # the usual serving batch: a million SIFT-shaped objects near 0.95 recall
        _search("search_million", 1_000_000, 128, 10_000, 10, 24),
        # wide rows scored in bf16 with the f32 re-rank of the final pool (GIST-shaped)
        _search("search_wide", 200_000, 960, 10_000, 10, 64, data="unit", cards="2/5/10/50",
                zipf=False, vec="bf16", rerank=True),
        # a heterogeneous batch: k of 1, 10 or 100 and ef of 16..512 per query
        dict(name="search_mixed", kind="batched", n=500_000, d=96, q=50_000, k=100, ef=512,
             data="float", comps=1000, cards="5/20/100", zipf=True, weights="constant",
             seeds="attribute"),
        # exact answers for a handful of queries (checking or small traffic)
        dict(name="brute_few", kind="brute", n=1_000_000, d=128, q=8, k=10, data="int",
             comps=1000, cards="3/10/20", zipf=True, weights="constant"),
        # the hybrid ground truth of a query set
        dict(name="brute_truth", kind="brute", n=1_000_000, d=128, q=10_000, k=10, data="int",
             comps=1000, cards="3/10/20", zipf=True, weights="filter"),
        # ground truth under the default weighting, k = 100, ragged sizes
        dict(name="brute_ragged", kind="brute", n=300_007, d=100, q=2_003, k=100, data="float",
             comps=1000, cards="5/20/100", zipf=True, weights="proportional"),
        # candidate sets of the default (f32) build
        dict(name="knn_f32", kind="knn", n=60_000, d=96, k=CANDIDATES, data="float", comps=500,
             cards="3/5/10", zipf=False, weights="proportional"),
        # raw vectors to a finished graph, as a serving index is made
        dict(name="build_million", kind="build", n=1_000_000, d=128, data="int", comps=1000,
             cards="3/10/20", zipf=True, weights="constant"),
        # the same on odd sizes of float rows with the default weighting
        dict(name="build_ragged", kind="build", n=120_011, d=100, data="float", comps=500,
             cards="3/5/10", zipf=False, weights="proportional"),
        # one training step of the learned entry point
        dict(name="entry_step", kind="entry", n=16_384, d=128, cells=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "batched", "brute", "brute", "knn", "build", "entry"])
    data = rng.choice(["int", "float"])
    cards, zipf = rng.choice([("3/10/20", True), ("3/5/10", False), ("5/20/100", True),
                              ("2/5/10/50", False)])
    weights = rng.choice(["constant", "proportional"])
    if kind == "search":
        n, d = _log(rng, 10_000, 1_000_000), _log(rng, 32, 960)
        n = min(n, 200_000_000 // d)
        if weights == "proportional":
            n = min(n, 250_000)
        k = rng.choice([1, 10, 100])
        vec = rng.choice(["f32", "f32", "bf16", "f16", "fp8"])
        if d > 256 or vec == "fp8":
            data = "unit"
        c = _search("", n, d, _log(rng, 1, 10_000), k, max(k, _log(rng, 16, 256)), data=data,
                    cards=cards, zipf=zipf, weights=weights, vec=vec, rerank=vec != "f32",
                    seeds=rng.choice(["attribute", "attribute", "nearest", "random"]))
        del c["name"]
        return c
    c = dict(kind=kind, data=data, comps=1000, cards=cards, zipf=zipf, weights=weights)
    if kind == "batched":
        c.update(n=_log(rng, 20_000, 250_000), d=rng.randint(64, 128), k=100, ef=512,
                 q=_log(rng, 500, 40_000), seeds="attribute")
    elif kind == "brute":
        d, n = _log(rng, 16, 960), _log(rng, 10_000, 1_000_000)
        n = min(n, 128_000_000 // d)
        c.update(n=n, d=d, q=min(_log(rng, 1, 10_000), 60_000_000_000 // (n * d)),
                 k=rng.choice([1, 10, 10, 100]),
                 weights=rng.choice(["constant", "proportional", "filter"]))
    elif kind == "knn":
        c.update(n=_log(rng, 5_000, 60_000), d=_log(rng, 32, 128), k=CANDIDATES, comps=500)
    elif kind == "build":
        c.update(n=_log(rng, 10_000, 1_000_000 if weights == "constant" else 120_000),
                 d=rng.randint(64, 128))
    else:
        return dict(kind="entry", n=_log(rng, 1_000, 16_384), d=rng.randint(64, 128),
                    cells=_log(rng, 64, 256))
    return c


# ------------------------------------------------------------------ inputs
def _rng(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _mixture(case, n, cent, g):
    """n points of the case's mixture, in slices."""
    d, k = case["d"], cent.shape[0]
    X = torch.empty((n, d), dtype=torch.float32, device=DEVICE)
    sigma = {"int": 20.0, "float": 0.3, "unit": 0.5}[case["data"]]
    for s in range(0, n, 1 << 17):
        e = min(n, s + (1 << 17))
        comp = torch.randint(0, k, (e - s,), generator=g, device=DEVICE)
        noise = torch.randn((e - s, d), generator=g, device=DEVICE)
        X[s:e] = cent[comp] + sigma * noise
    if case["data"] == "int":
        X.round_().clamp_(0, 255)
    elif case["data"] == "unit":
        X /= X.norm(dim=1, keepdim=True)
    return X


def _cards(case):
    return [int(c) for c in case["cards"].split("/")]


def _probabilities(case, card):
    p = 1.0 / torch.arange(1, card + 1, dtype=torch.float64)
    p = p if case["zipf"] else torch.ones(card, dtype=torch.float64)
    return p / p.sum()


def _attributes(case, n, g):
    cols = []
    for card in _cards(case):
        edge = _probabilities(case, card).cumsum(0)[:-1].to(DEVICE)
        u = torch.rand(n, generator=g, device=DEVICE, dtype=torch.float64)
        cols.append(torch.bucketize(u, edge, right=True).to(torch.uint8))
    return torch.stack(cols, dim=1).contiguous()


def _inputs(case, seed):
    """Objects, queries and their attributes (queries absent for knn and build)."""
    g = _rng(seed)
    cent = torch.randn((case["comps"], case["d"]), generator=g, device=DEVICE)
    if case["data"] == "int":
        cent = (64.0 + 40.0 * cent).round().clamp(0, 255)
    X = _mixture(case, case["n"], cent, g)
    A = _attributes(case, case["n"], g)
    if "q" not in case:
        return X, A, None, None
    return X, A, _mixture(case, case["q"], cent, g), _attributes(case, case["q"], g)


def _index_weights(case):
    return (1.0, 10000.0) if case["weights"] == "constant" else None


def _entry_inputs(case, seed):
    g = _rng(seed)
    d, E, n = case["d"], case["cells"], case["n"]
    cent = torch.randn((E, d), generator=g, device=DEVICE)
    y = torch.randint(0, E, (n,), generator=g, device=DEVICE)
    Q = cent[y] + 0.3 * torch.randn((n, d), generator=g, device=DEVICE)
    P = 0.05 * torch.randn(nhq.nhq_entry_param_count(d, E), generator=g, device=DEVICE)
    P[0] = 1.0 / math.sqrt(1.09 * d)  # the input scale: rows of about unit norm
    return P, Q, y.to(torch.int32)


def _outputs(q, k):
    return {"ids": torch.empty((q, k), dtype=torch.uint32, device=DEVICE),
            "dists": torch.empty((q, k), dtype=torch.float32, device=DEVICE),
            "chi": torch.empty((q, k), dtype=torch.uint8, device=DEVICE)}


def prepare(case, seed):
    s = {"case": case}
    kind = case["kind"]
    if kind == "entry":
        s["P"], s["Q"], s["y"] = _entry_inputs(case, seed)
        s["out"] = {"grad": torch.empty_like(s["P"]),
                    "loss": torch.empty(1, dtype=torch.float32, device=DEVICE)}
        return s
    X, A, Q, QA = _inputs(case, seed)
    if kind == "build":
        s.update(X=X, A=A)
        s["out"] = {"graph": torch.empty((case["n"], DEGREE), dtype=torch.uint32,
                                         device=DEVICE)}
        return s
    if kind in ("search", "batched"):
        s["index"] = nhq.Index.build(X, A, degree=DEGREE, weights=_index_weights(case),
                                     K=CANDIDATES, knn_dtype=1)
    else:
        s["index"] = nhq.Index.create(X, A, _index_weights(case))
    if kind == "knn":
        s["out"] = {"ids": torch.empty((case["n"], case["k"]), dtype=torch.uint32,
                                       device=DEVICE),
                    "dists": torch.empty((case["n"], case["k"]), dtype=torch.float32,
                                         device=DEVICE)}
        return s
    s.update(Q=Q, QA=QA, out=_outputs(case["q"], case["k"]))
    if kind == "batched":
        g = _rng(seed + 1_000_003)
        pick = torch.randint(0, 3, (case["q"],), generator=g, device=DEVICE)
        s["k"] = torch.tensor([1, 10, 100], dtype=torch.int32, device=DEVICE)[pick]
        lo = s["k"].clamp(min=16).to(torch.float32)
        u = torch.rand(case["q"], generator=g, device=DEVICE)
        s["ef"] = (lo + (u * (case["ef"] - lo + 1)).floor()).clamp(max=case["ef"]).to(torch.int32)
    return s


def run(state):
    case, out = state["case"], state["out"]
    kind = case["kind"]
    if kind == "search":
        nhq.nhq_search(state["index"].handle, state["Q"], state["QA"], case["k"], case["ef"],
                       out["ids"], out["dists"], out["chi"], seed=1,
                       vec_dtype=VEC[case["vec"]], rerank=int(case["rerank"]),
                       seed_mode=SEEDS[case["seeds"]])
    elif kind == "batched":
        nhq.nhq_search_batched(state["index"].handle, state["Q"], state["QA"], state["k"],
                               state["ef"], case["k"], out["ids"], out["dists"], out["chi"],
                               seed=1, seed_mode=SEEDS[case["seeds"]])
    elif kind == "brute":
        weights = "filter" if case["weights"] == "filter" else "index"
        nhq.nhq_brute_force(state["index"].handle, state["Q"], state["QA"], case["k"],
                            out["ids"], out["dists"], out["chi"], weights=weights)
    elif kind == "knn":
        nhq.nhq_knn(state["index"].handle, case["k"], out["ids"], out["dists"])
    elif kind == "build":
        with nhq.Index.build(state["X"], state["A"], degree=DEGREE,
                             weights=_index_weights(case), K=CANDIDATES, knn_dtype=1) as ix:
            nhq.nhq_index_get_graph(ix.handle, out["graph"])
    else:
        nhq.nhq_entry_grad(state["P"], case["cells"], state["Q"], state["y"], out["grad"],
                           out["loss"])
    # ids as signed integers, which torch can index and compare
    return {name: t.view(torch.int32) if t.dtype == torch.uint32 else t
            for name, t in out.items()}


# ------------------------------------------------------------------ work and exact values
def _share(case):
    """Share of all pairs whose distance matters: under constant and filter weights the
    objects that carry the query's tuple."""
    if case["weights"] == "proportional":
        return 1.0
    return math.prod(float((_probabilities(case, c) ** 2).sum()) for c in _cards(case))


def work(case):
    d, n, kind = case["d"], case["n"], case["kind"]
    if kind == "entry":
        E = case["cells"]
        params = 1 + d * 64 + 64 + 64 * E + E
        # forward and weight gradients of both layers, and the hidden gradient
        return {"bytes": 4.0 * (n * (d + 1) + 2 * params + 1),
                "flops": 2.0 * n * (2 * d * 64 + 3 * 64 * E)}
    m = len(_cards(case))
    if kind == "build":
        return {"bytes": float(n * (4 * d + m + 4 * DEGREE)),
                "flops": 2.0 * n * n * d * _share(case)}
    if kind == "knn":
        return {"bytes": float(n * (4 * d + m + 8 * case["k"])),
                "flops": 2.0 * n * n * d * _share(case)}
    q, k = case["q"], case["k"]
    io = q * (4.0 * d + m + 9 * k)
    if kind == "brute":
        return {"bytes": io + n * (4.0 * d + m), "flops": 2.0 * q * n * d * _share(case)}
    # a search expands about ef records (264 on average in the mixed batch), reads each
    # one's adjacency and neighbour attributes, and evaluates about 15 rows for each
    expanded = q * (case["ef"] if kind == "search" else 0.5 * case["ef"] + 8)
    size = {"f32": 4, "bf16": 2, "f16": 2, "fp8": 1}[case.get("vec", "f32")]
    rows = min(15.0 * expanded, float(q) * n)
    return {"bytes": io + expanded * 8 * DEGREE + rows * d * size, "flops": 3.0 * rows * d}


def _fused(case, q, QA, X, A, X2, filtered):
    """Gamma of query rows q against every object, in 64 bits."""
    delta = (q.square().sum(1, keepdim=True) + X2 - 2.0 * (q @ X.T)).clamp_(min=0).sqrt_()
    chi = torch.zeros(delta.shape, dtype=torch.uint8, device=DEVICE)
    for j in range(A.shape[1]):
        chi += QA[:, j, None] != A[None, :, j]
    if filtered:
        return delta.masked_fill_(chi > 0, math.inf)
    if case["weights"] == "constant":
        return delta.add_(chi.double(), alpha=10000.0)
    return delta.mul_(1.0 + chi.double() / A.shape[1])


def exact(case, seed):
    kind = case["kind"]
    if kind == "entry":
        return _exact_entry(case, seed)
    if kind not in ("brute", "knn"):
        return None  # the answer depends on the graph
    X, A, Q, QA = _inputs(case, seed)
    X = X.double()
    if kind == "knn":
        Q, QA = X, A
    X2 = X.square().sum(1)[None, :]
    rows = max(1, 200_000_000 // X.shape[0])
    dists = []
    for s in range(0, Q.shape[0], rows):
        g = _fused(case, Q[s:s + rows].double(), QA[s:s + rows], X, A, X2,
                   case["weights"] == "filter")
        if kind == "knn":
            i = torch.arange(g.shape[0], device=DEVICE)
            g[i, s + i] = math.inf
        dists.append(g.topk(min(case["k"], g.shape[1]), dim=1, largest=False).values)
    return {"ids": None, "dists": torch.cat(dists), "chi": None}


def _exact_entry(case, seed):
    P, Q, y = _entry_inputs(case, seed)
    d, E = case["d"], case["cells"]
    P = P.double().requires_grad_(True)
    w1, b1 = P[1:1 + 64 * d].view(d, 64), P[1 + 64 * d:65 + 64 * d]
    w2, b2 = P[65 + 64 * d:65 + 64 * (d + E)].view(64, E), P[65 + 64 * (d + E):]
    x = Q.double() * P[0].detach()
    loss = torch.nn.functional.cross_entropy(torch.relu(x @ w1 + b1) @ w2 + b2, y.long())
    loss.backward()
    return {"grad": P.grad, "loss": loss.detach().view(1)}
