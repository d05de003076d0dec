"""What this library is measured on: the calls a user makes, over the sizes they are made at.

A case is one call (or one call and its read-out) of the public Python entry points on synthetic
SPLADE-shaped data drawn on the GPU: 64 latent topics, each a Zipf(1) law over its own permutation of a
30,522-term vocabulary, a Dirichlet(0.1) topic mixture per row, distinct terms, values
|N(0, 1)| * (1 + exp(-rank / 20)).  Documents hold about 120 entries (10..400), queries 10..150.

The collection of a search case is fixed and its index is built once per process (a program that serves
queries keeps its index); the queries, requests and training rows come from the seed.  Cases that build
something draw the documents from the seed too.

Collections:
  "100k"   100,000 documents, lists of 2,000, 100 blocks a list, fp32 summaries, unpruned lists kept
  "300k16" 300,000 documents, lists of 6,000, 400 blocks, u8 summaries, 16-bit forward values
  "1M"     1,000,000 documents, lists of 6,000, 400 blocks, u8 summaries; a 10-neighbour graph and a
           parameter network where a case uses them
  "small"  a drawn number of documents, list length and block count (u8 or fp32 summaries)
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2509_24815_gb300 as sz

VOCAB = 30522
TOPICS = 64
KAPPA = 10
COLLECTIONS = {
    "100k": dict(n_docs=100_000, lam=2000, beta=100, u8=False, fp16=False, full=True),
    "300k16": dict(n_docs=300_000, lam=6000, beta=400, u8=True, fp16=True, full=False),
    "1M": dict(n_docs=1_000_000, lam=6000, beta=400, u8=True, fp16=False, full=False),
}


# --------------------------------------------------------------------------- cases
def _search(name, on, nq, cut, hf, *, k=10, wave=1, persistent=False, host=False, long=True, exhaustive=False,
            use_knn=False, learned=False, **small):
    return dict(name=name, kind="search", on=on, nq=nq, cut=cut, hf=hf, k=k, wave=wave, persistent=persistent,
                host=host, long=long, exhaustive=exhaustive, use_knn=use_knn, learned=learned, **small)


def listed():
    return [
        # an interactive lookup: one query, the default parameters, buffers on the device
        _search("one query", "1M", 1, 10, 0.8),
        # the README's call: numpy queries in, numpy results out, default parameters
        _search("host batch", "100k", 1000, 10, 0.8, host=True, long=False),
        # every block of the query's lists visited (rank-exact on the pruned lists; quality checks, ground truth)
        _search("exhaustive", "100k", 1000, 10, 0.8, long=False, exhaustive=True),
        # the batched configuration in its tuned launch: offline scoring of a query log
        _search("batch", "1M", 10_000, 10, 0.8, wave=8, persistent=True),
        # the same on an index with 16-bit forward values (the compact form), a ragged batch
        _search("batch 16-bit", "300k16", 4999, 5, 0.9, wave=8, persistent=True),
        # the high-recall operating point with the neighbour-graph expansion
        _search("graph", "1M", 10_000, 30, 0.9, wave=4, persistent=True, use_knn=True),
        # per-query learned (cut, heap_factor), a deep result list (re-ranking), an odd batch
        _search("learned top 100", "1M", 2047, 10, 0.8, k=100, wave=8, persistent=True, learned=True),
        # exact top-k by brute force: the recall judge, and the labels of the learned parameters
        dict(name="exact", kind="exact", on="100k", nq=1000, k=10, long=False),
        # continuous batching: requests of mixed length and k arriving faster than they are served
        dict(name="serve", kind="serve", on="1M", n=4096, rate=200_000, cut=5, hf=0.9, max_batch=1024, streams=16),
        # one training step (forward, backward, Adam) of the parameter network at its training batch size
        dict(name="train step", kind="train", n=4096),
        # indexing a collection from host memory
        dict(name="build", kind="build", n_docs=100_000, lam=2000, beta=100, u8=True, fp16=False),
        # the neighbour graph of a collection: by search, then one refinement pass
        dict(name="neighbour graph", kind="knn", n_docs=20_000, lam=2000, beta=100, cut=10, hf=0.9),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 7 + ["exact", "serve", "train", "build", "knn"])
    if kind == "search":
        on = rng.choice(["100k", "300k16", "1M", "small"])
        c = _search("", on, _log(rng, 1, 10_000), _log(rng, 3, 30), round(rng.uniform(0.5, 1.0), 3),
                    k=_log(rng, 1, 128), wave=rng.choice([1, 1, 4, 8, 16]), persistent=rng.random() < 0.6,
                    host=rng.random() < 0.3, long=rng.random() < 0.7)
        del c["name"]
        if on == "small":
            c.update(n_docs=_log(rng, 2_000, 100_000), lam=_log(rng, 150, 4000), beta=_log(rng, 12, 300),
                     u8=rng.random() < 0.5)
            c["exhaustive"] = rng.random() < 0.3
        elif on == "1M":
            c["use_knn"] = rng.random() < 0.4
            c["learned"] = rng.random() < 0.25
        if c["exhaustive"] or not c["persistent"]:  # as costly a pass as the largest listed case at most
            c["nq"] = max(1, min(c["nq"], 2000))
            c["cut"] = min(c["cut"], 15)
        return c
    if kind == "exact":
        return dict(kind="exact", on="100k", nq=_log(rng, 1, 1000), k=_log(rng, 1, 200), long=rng.random() < 0.4)
    if kind == "serve":
        return dict(kind="serve", on=rng.choice(["300k16", "1M"]), n=_log(rng, 500, 4096),
                    rate=_log(rng, 20_000, 400_000), cut=rng.randint(3, 10), hf=round(rng.uniform(0.8, 1.0), 3),
                    max_batch=rng.choice([256, 1024]), streams=rng.choice([4, 16]))
    if kind == "train":
        return dict(kind="train", n=_log(rng, 100, 20_000))
    if kind == "build":
        return dict(kind="build", n_docs=_log(rng, 5_000, 100_000), lam=_log(rng, 200, 2000), beta=_log(rng, 16, 100),
                    u8=rng.random() < 0.6, fp16=rng.random() < 0.4)
    return dict(kind="knn", n_docs=_log(rng, 3_000, 20_000), lam=_log(rng, 300, 2000), beta=_log(rng, 16, 100),
                cut=rng.randint(4, 12), hf=round(rng.uniform(0.8, 1.0), 3))


# --------------------------------------------------------------------------- data
_model = None


def _topics():
    """(perm [TOPICS, VOCAB], Zipf cumulative table): one topic model for documents and queries."""
    global _model
    if _model is None:
        g = torch.Generator(device="cuda").manual_seed(20250924)
        perm = torch.rand((TOPICS, VOCAB), generator=g, device="cuda").argsort(dim=1)
        mass = 1.0 / torch.arange(1, VOCAB + 1, device="cuda", dtype=torch.float64)
        _model = perm, torch.cumsum(mass / mass.sum(), 0).float()
    return _model


def _rows(n, seed, stream, lens):
    """n rows as device CSR pieces (indptr int64, terms int16, vals float32), terms ascending and distinct.
    Each row draws topic-first, rank-second and keeps its first `lens` distinct terms."""
    perm, cdf = _topics()
    terms, vals, counts = [], [], []
    step = 32768
    for at in range(0, n, step):
        m = min(step, n - at)
        g = torch.Generator(device="cuda").manual_seed((seed * 16 + stream) * 4096 + at // step)
        want = lens(m, g)
        width = 512  # draws per row: enough distinct terms but for the longest rows, which keep what they got
        mix = torch._standard_gamma(torch.full((m, TOPICS), 0.1, device="cuda", dtype=torch.float64), generator=g)
        cum = torch.cumsum((mix + 1e-300) / (mix + 1e-300).sum(1, keepdim=True), 1).float()
        topic = torch.searchsorted(cum, torch.rand((m, width), generator=g, device="cuda")).clamp_(max=TOPICS - 1)
        rank = torch.searchsorted(cdf, torch.rand((m, width), generator=g, device="cuda")).clamp_(max=VOCAB - 1)
        key = (perm[topic, rank] * width + torch.arange(width, device="cuda")).int().sort(dim=1).values
        term, pos = key // width, (key % width).long()
        first = torch.ones_like(term, dtype=torch.bool)
        first[:, 1:] = term[:, 1:] != term[:, :-1]
        order = torch.zeros_like(term).scatter_(1, pos, first.int()).cumsum(1).gather(1, pos)
        keep = first & (order <= want[:, None])
        x = torch.randn((m, width), generator=g, device="cuda").abs_().clamp_(min=1e-6)
        v = x * (1.0 + torch.exp(-rank.gather(1, pos).float() / 20.0))
        terms.append(term[keep].short())
        vals.append(v[keep].float())
        counts.append(keep.sum(1))
    indptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    indptr[1:] = torch.cumsum(torch.cat(counts), 0)
    return indptr, torch.cat(terms), torch.cat(vals)


def _lognormal(mean, sd, lo, hi):
    s2 = math.log(1.0 + sd * sd / (mean * mean))
    mu = math.log(mean) - 0.5 * s2
    return lambda m, g: torch.exp(mu + math.sqrt(s2) * torch.randn(m, generator=g, device="cuda")).round().clamp(lo, hi).int()


def _uniform(lo, hi):
    return lambda m, g: torch.randint(lo, hi + 1, (m,), generator=g, device="cuda", dtype=torch.int32)


def _documents(n, seed):
    return _rows(n, seed, 1, _lognormal(120.0, 40.0, 10, 400))


def _queries(n, seed, long):
    return _rows(n, seed, 2, _uniform(10, 150) if long else _lognormal(40.0, 15.0, 10, 150))


def _host(rows):
    ip, t, v = rows
    return SimpleNamespace(indptr=ip.cpu().numpy().astype(np.uint64), terms=t.cpu().numpy().view(np.uint16),
                           vals=v.cpu().numpy(), dim=VOCAB)


def _device(rows):
    ip, t, v = rows
    return sz.DeviceCSR(ip, t, v, VOCAB, int((ip[1:] - ip[:-1]).max()))


# --------------------------------------------------------------------------- indexes
_kept = {}  # the last few indexes, by what they are built from


def _spec(case):
    if case["on"] == "small":
        return dict(n_docs=case["n_docs"], lam=case["lam"], beta=case["beta"], u8=case["u8"], fp16=False, full=False)
    return COLLECTIONS[case["on"]]


def _build(docs, c):
    return sz.seismic_build(docs, lambda_=c["lam"], beta=c["beta"], alpha=0.4, quantize_u8=c["u8"], seed=0,
                            keep_full_lists=c.get("full", False), values_fp16=c["fp16"])


def _mlp_weights():
    """A fixed parameter network whose predictions differ from query to query."""
    g = np.random.default_rng(5)
    w1 = g.standard_normal((128, 64)) * np.sqrt(2.0 / 64) / 8
    w2 = g.standard_normal((64, 128)) * np.sqrt(2.0 / 128)
    w3 = g.standard_normal((2, 64)) * 0.2
    return np.concatenate([w1.ravel(), np.zeros(128), w2.ravel(), np.zeros(64), w3.ravel(), [-1.0, 0.5]]).astype(np.float32)


def _index(case):
    c = _spec(case)
    key = tuple(sorted(c.items()))
    if key not in _kept:
        while len(_kept) >= 4:
            _kept.pop(next(iter(_kept)))
        _kept[key] = _build(_device(_documents(c["n_docs"], 0)), c)
    ix = _kept[key]
    if case.get("use_knn") and not ix.info()["kappa"]:
        sz.seismic_build_knn(ix, KAPPA, sz.search_params(cut=3, heap_factor=1.0, wave=8, persistent=True))
    if case.get("learned") and not ix.info()["has_mlp"]:
        sz.seismic_set_mlp(ix, _mlp_weights())
    return ix


# --------------------------------------------------------------------------- the three calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        g = torch.Generator(device="cuda").manual_seed(seed)
        w = torch.from_numpy(_mlp_weights()).cuda()
        n = case["n"]
        feat = torch.zeros((n, sz.MLP_IN), device="cuda")
        feat[:, :51] = torch.rand((n, 51), generator=g, device="cuda") * 4.0
        feat[:, 49:51] *= torch.tensor([25.0, 4.0], device="cuda")  # the L1 and L2 norms
        # as in the middle of a training run: moments of earlier steps, step 200
        return dict(kind=kind, w=w, g=torch.zeros_like(w), step=200,
                    m=torch.randn(w.shape, generator=g, device="cuda") * 1e-3,
                    v=torch.rand(w.shape, generator=g, device="cuda") * 1e-5 + 1e-6, feat=feat,
                    tgt=torch.rand((n, 2), generator=g, device="cuda"), loss=torch.zeros(1, device="cuda"))
    if kind == "build":
        return dict(kind=kind, docs=_host(_documents(case["n_docs"], seed + 1)), case=case,
                    q=_device(_queries(256, seed + 1, False)))
    if kind == "knn":
        c = dict(lam=case["lam"], beta=case["beta"], u8=True, fp16=False)
        return dict(kind=kind, ix=_build(_device(_documents(case["n_docs"], seed + 1)), c),
                    params=sz.search_params(cut=case["cut"], heap_factor=case["hf"], wave=8, persistent=True))
    ix = _index(case)
    if kind == "exact":
        return dict(kind=kind, ix=ix, q=_device(_queries(case["nq"], seed, case["long"])), k=case["k"])
    if kind == "serve":
        n = case["n"]
        rng = np.random.default_rng(seed)
        params = sz.search_params(cut=case["cut"], heap_factor=case["hf"], wave=8, persistent=True)
        return dict(kind=kind, q=_host(_queries(n, seed, True)),
                    at=np.cumsum(rng.exponential(1.0 / case["rate"], size=n)),
                    k=rng.choice(np.array([10, 100], dtype=np.uint32), size=n, p=[0.9, 0.1]),
                    srv=sz.Server(ix, params, max_batch=case["max_batch"], streams=case["streams"], max_query_nnz=160))
    rows = _queries(case["nq"], seed, case["long"])
    params = sz.search_params(k=case["k"], cut=case["cut"], heap_factor=case["hf"], wave=case["wave"],
                              persistent=case["persistent"], exhaustive=case["exhaustive"], use_knn=case["use_knn"],
                              learned=case["learned"])
    return dict(kind=kind, ix=ix, q=_host(rows) if case["host"] else _device(rows), params=params)


def _padded(a, n):
    """An exported array, whose length depends on the documents, in an array of its largest length."""
    out = np.zeros(n, dtype=np.int32 if a.dtype.kind == "u" else a.dtype)
    out[:len(a)] = a.view(out.dtype)
    return out


def run(state):
    kind = state["kind"]
    if kind == "search":
        ids, scores = sz.seismic_search(state["ix"], state["q"], state["params"])
        return ids.view(np.int32) if isinstance(ids, np.ndarray) else ids, scores
    if kind == "exact":
        return sz.seismic_search_exact(state["ix"], state["q"], state["k"])
    if kind == "serve":
        ids, scores, _, _ = state["srv"].replay(state["q"], state["at"], state["k"])
        return ids.view(np.int32), scores
    if kind == "train":
        state["step"] += 1
        sz.seismic_mlp_train_step(state["w"], state["g"], state["m"], state["v"], state["feat"], state["tgt"], 2e-3,
                                  state["step"], state["loss"])
        return dict(w=state["w"], g=state["g"], m=state["m"], v=state["v"], loss=state["loss"])
    if kind == "build":  # the index's blocks read back, and a first search on it
        c = state["case"]
        ix = _build(state["docs"], c)
        ids, scores = sz.seismic_search(ix, state["q"], sz.search_params(cut=10, heap_factor=0.8))
        blocks, posts = VOCAB * c["beta"], min(VOCAB * c["lam"], 128 * c["n_docs"])
        out = {n: _padded(sz.seismic_export(ix, n), cap)
               for n, cap in (("list_ptr", VOCAB + 1), ("blk_ptr", VOCAB + 1), ("bdoc_ptr", blocks + 1), ("bdoc", posts),
                              ("blk_m", blocks), ("blk_size", blocks))}
        ix.close()
        return dict(out, ids=ids, scores=scores)
    sz.seismic_build_knn(state["ix"], KAPPA, state["params"])
    sz.seismic_refine_knn(state["ix"], 1)
    return sz.seismic_get_knn(state["ix"]).view(np.int32)


_worked = {}


def work(case):
    """Searches: each entry of a batch's own work counted by the search itself -- the rows, summary columns
    and block members the method has to look at for these queries -- but no more than the arrays of the index
    that search reads, once, since queries of a batch may share them.  Two operations for each summary entry
    and each entry of a scored row."""
    kind = case["kind"]
    if kind == "train":
        p = sz.MLP_PARAMS
        return {"bytes": 4 * (7 * p + case["n"] * (sz.MLP_IN + 2)), "flops": 6 * case["n"] * p}
    key = repr(sorted(case.items()))
    if key not in _worked:
        _worked[key] = _count(case)
    return _worked[key]


def _count(case):
    kind = case["kind"]
    if kind in ("build", "knn"):
        n, rows = case["n_docs"], _documents(case["n_docs"], 1)
        nnz = int(rows[0][-1])
        sizes = torch.bincount(rows[1].long(), minlength=VOCAB).clamp(max=case["lam"])
        posts, row = int(sizes.sum()), nnz / n
        if kind == "build":  # documents in, lists and blocks out; every member against its list's centroids
            return {"bytes": 6 * nnz + 6 * nnz + 24 * posts, "flops": 2 * posts * row * 2}
        # every row in, the graph out; a query's lists hold about lam members, a tenth of them scored
        return {"bytes": 6 * nnz + 4 * n * KAPPA, "flops": 2 * n * row * (case["cut"] * case["lam"] / 10 + KAPPA * KAPPA)}
    if kind == "exact":
        rows = _documents(COLLECTIONS[case["on"]]["n_docs"], 0)
        nnz, df = int(rows[0][-1]), torch.bincount(rows[1].long(), minlength=VOCAB)
        q = _queries(case["nq"], 1, case["long"])
        return {"bytes": min(8 * nnz, 8 * int(df[q[1].long()].sum())) + 8 * case["nq"] * case["k"],
                "flops": 2 * int(df[q[1].long()].sum())}
    c = dict(case)
    if kind == "serve":
        c.update(kind="search", nq=case["n"], long=True, k=10, wave=8, persistent=True, host=False, exhaustive=False,
                 use_knn=False, learned=False)
    s = prepare(c, 1)
    q = s["q"] if isinstance(s["q"], sz.DeviceCSR) else _device(_queries(c["nq"], 1, c["long"]))
    st = sz.seismic_search(s["ix"], q, s["params"], stats=True)[2].astype(np.float64).sum(0)
    n = dict(zip(sz.STATS, st))
    info = s["ix"].info()
    entry, code = (4 if info["values_fp16"] else 6), (3 if info["quantize_u8"] else 6)
    touched = (6 * n["query_nnz"] + 4 * n["dir_lookups"] + code * n["summary_entries"] + 8 * n["blocks_scored"]
               + 4 * n["block_docs"] + 8 * n["docs"] + entry * (n["doc_nnz"] + n["knn_nnz"]) + 8 * n["knn_docs"])
    once = (entry * info["nnz"] + 12 * info["n_postings"] + code * info["n_summary_entries"] + 8 * info["n_blocks"]
            + 6 * n["query_nnz"])
    return {"bytes": min(touched, once) + 8 * c["nq"] * c["k"],
            "flops": 2 * (n["summary_entries"] + n["doc_nnz"] + n["knn_nnz"])}


# --------------------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """fp64 values where the result is defined without the index's clustering: exact search, exhaustive
    traversal (the best of the documents in the query's pruned lists) and the training step.  What a pruned
    search returns depends on the clusters, and an index is whole numbers: None."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "exact" or (case["kind"] == "search" and case["exhaustive"]):
        return [None, _exact_scores(case, seed)]
    return None


def _sparse(ip, cols, vals):
    return torch.sparse_csr_tensor(ip, cols, vals, size=(ip.numel() - 1, VOCAB))


def _exact_scores(case, seed):
    c = _spec(case)
    ip, t, v = _documents(c["n_docs"], 0)
    t = t.long()
    docs = _sparse(ip, t, v.double())
    qip, qt, qv = _queries(case["nq"], seed, case["long"])
    qrow = torch.repeat_interleave(torch.arange(case["nq"], device="cuda"), qip[1:] - qip[:-1])
    member = None
    if case["kind"] == "search":  # list t: the lam largest values of term t, earlier documents first on ties
        by = torch.sort(v, descending=True, stable=True).indices
        by = by[torch.sort(t[by], stable=True).indices]
        start = torch.searchsorted(t[by].contiguous(), torch.arange(VOCAB, device="cuda"))
        rank = torch.empty_like(t)
        rank[by] = torch.arange(t.numel(), device="cuda") - start[t[by]]
        member = _sparse(ip, t, (rank < c["lam"]).double())
        by = torch.sort(qv, descending=True, stable=True).indices  # the query's `cut` largest terms
        by = by[torch.sort(qrow[by], stable=True).indices]
        place = torch.empty_like(qrow)
        place[by] = torch.arange(qrow.numel(), device="cuda") - qip[qrow[by]]
    out = []
    for a in range(0, case["nq"], 128):
        b = min(case["nq"], a + 128)
        sel = (qrow >= a) & (qrow < b)
        dense = torch.zeros((VOCAB, b - a), dtype=torch.float64, device="cuda")
        dense[qt[sel].long(), qrow[sel] - a] = qv[sel].double()
        score = docs @ dense
        if member is not None:
            dense.zero_()
            use = sel & (place < case["cut"])
            dense[qt[use].long(), qrow[use] - a] = 1.0
            score = torch.where((member @ dense) > 0.0, score, torch.full_like(score, -math.inf))
        k = min(case["k"], score.shape[0])
        top = torch.full((b - a, case["k"]), -math.inf, dtype=torch.float64, device="cuda")
        top[:, :k] = torch.topk(score, k, dim=0).values.t()
        out.append(top)
    return torch.cat(out)


def _exact_train(case, seed):
    s = prepare(case, seed)
    w, feat, tgt, n, step = s["w"].double(), s["feat"], s["tgt"].double(), case["n"], s["step"] + 1

    def bf16(x):
        return x.bfloat16().double()

    cuts = np.cumsum([0, 128 * 64, 128, 64 * 128, 64, 2 * 64, 2])
    w1, b1, w2, b2, w3, b3 = (w[cuts[i]:cuts[i + 1]] for i in range(6))
    w1, w2, w3 = w1.view(128, 64), w2.view(64, 128), w3.view(2, 64)
    a0 = bf16(feat)
    z1 = a0 @ w1.t() + b1
    a1 = bf16(z1.clamp(min=0))
    z2 = a1 @ w2.t() + b2
    a2 = bf16(z2.clamp(min=0))
    sg = torch.sigmoid(a2 @ w3.t() + b3)
    e = sg - tgt
    do = 2.0 * e * sg * (1.0 - sg) / n
    d2 = (do @ w3) * (z2 > 0)
    d1 = (d2 @ w2) * (z1 > 0)
    g = torch.cat([(d1.t() @ a0).reshape(-1), d1.sum(0), (d2.t() @ a1).reshape(-1), d2.sum(0), (do.t() @ a2).reshape(-1), do.sum(0)])
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    new = w - 2e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return dict(w=new, g=g, m=m, v=v, loss=(e * e).sum().reshape(1) / n)
