"""Calls at the sizes where a kernel takes another route: each against an exact reference computed here, or against
the route that the same call takes under other launch parameters."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _rows(n, terms_of, vlo, vhi, dim, rng):
    """n sparse rows of small whole values (fp32 sums of products are exact, and ties are common); terms_of(i) gives
    row i's terms."""
    t = [np.unique(terms_of(i)) for i in range(n)]
    indptr = np.zeros(n + 1, dtype=np.uint64)
    np.cumsum([len(x) for x in t], out=indptr[1:])
    vals = rng.integers(vlo, vhi + 1, int(indptr[-1]))
    vals[vals == 0] = 1
    return synth.CSR(indptr, np.concatenate(t).astype(np.uint16), vals.astype(np.float32), dim)


def _scores(queries, docs):
    sp = pytest.importorskip("scipy.sparse")

    def csr(m):
        return sp.csr_matrix((m.vals.astype(np.float64), m.terms.astype(np.int64), m.indptr.astype(np.int64)),
                             shape=(m.n_rows, m.dim))
    return (csr(queries) @ csr(docs).T).toarray()


# Exact search: tiles of 24,576 documents up to k = 256, of 16,384 past it, and as many CTAs per query as run at once.
@pytest.mark.parametrize("n_docs", [24576, 24577, 49153])
@pytest.mark.parametrize("nq,k", [(1, 256), (1, 257), (150, 10), (310, 256)])
def test_exact_search_tile_edges(sz, n_docs, nq, k):
    dim = 61
    rng = np.random.default_rng(n_docs + k)
    docs = _rows(n_docs, lambda i: rng.integers(0, dim, rng.integers(1, 6)), -2, 5, dim, rng)
    queries = _rows(nq, lambda i: rng.integers(0, dim, rng.integers(1, 40)), -1, 3, dim, rng)
    ix = sz.seismic_build(docs, lambda_=10, beta=2, alpha=0.5, seed=1, keep_full_lists=True)
    ids, sc = sz.seismic_search_exact(ix, queries, k)
    ix.close()
    score = _scores(queries, docs)
    order = np.argsort(-score, axis=1, kind="stable")[:, :k]  # score descending, id ascending
    np.testing.assert_array_equal(ids, order.astype(np.uint32))
    np.testing.assert_array_equal(sc, np.take_along_axis(score, order, 1).astype(np.float32))


# Exact search: a tile (24,576 documents, 16,384 past k = 256) without a posting of the query is passed over and one
# with few of them offers only those, once documents of score 0 cannot enter any more.  Queries of one rare term, of
# some (their offers wait over several tiles) and of many and common ones; negative scores, which rank behind 0.
@pytest.mark.parametrize("n_docs", [24577, 70003])
@pytest.mark.parametrize("nq,k", [(1, 1), (3, 10), (400, 10), (400, 256), (700, 3), (40, 257), (400, 1000)])
def test_exact_search_of_rare_terms(sz, n_docs, nq, k):
    dim = 3000
    rng = np.random.default_rng(n_docs + k)
    docs = _rows(n_docs, lambda i: np.concatenate([rng.integers(0, 4, 1), rng.integers(4, dim, rng.integers(1, 4))]), -2, 5,
                 dim, rng)
    sizes = [1, 1, 2, 7, 25, 60, 600]
    queries = _rows(nq, lambda i: rng.integers(4 if i % 5 else 0, dim, sizes[i % 7]), -1 if nq > 1 else 1, 3, dim, rng)
    ix = sz.seismic_build(docs, lambda_=10, beta=2, alpha=0.5, seed=1, keep_full_lists=True)
    ids, sc = sz.seismic_search_exact(ix, queries, k)
    ix.close()
    score = _scores(queries, docs)
    order = np.argsort(-score, axis=1, kind="stable")[:, :k]  # score descending, id ascending
    np.testing.assert_array_equal(ids, order.astype(np.uint32))
    np.testing.assert_array_equal(sc, np.take_along_axis(score, order, 1).astype(np.float32))


@pytest.fixture(scope="module", params=[False, True], ids=["fp32", "fp16"])
def collection(sz, request):
    """3000 rows of 1..60 of 300 terms, some of them longer than a queue's positions, and a graph."""
    dim = 4000
    rng = np.random.default_rng(3)
    docs = _rows(3000, lambda i: rng.integers(0, dim, 3500) if i % 500 == 7 else rng.integers(0, 300, rng.integers(1, 61)),
                 -1, 4, dim, rng)
    queries = _rows(1400, lambda i: rng.integers(0, 320, rng.integers(1, 90)), -1, 3, dim, rng)
    ix = sz.seismic_build(docs, lambda_=300, beta=40, alpha=0.6, quantize_u8=False, seed=2, values_fp16=request.param)
    sz.seismic_set_knn(ix, rng.integers(0, docs.n_rows, (docs.n_rows, 5)))
    yield queries, ix
    ix.close()


# The default launch (group 1) by the number of queries: CTAs of 32, 16 and 8 warps, five CTAs of 8 warps per SM;
# waves are scored together from the first full top-k on.  Lane groups score one row and one wave at a time; sums of
# whole values are exact in any order, so the documents, the scores and the work counted have to be the same.
@pytest.mark.parametrize("kw", [dict(wave=1), dict(wave=1, k=70, heap_factor=1.0), dict(wave=8, k=100), dict(wave=8, use_knn=True),
                                dict(wave=3, hf_mode=1, heap_factor=0.9), dict(exhaustive=True), dict(wave=2, cta_warps=8)],
                         ids=lambda d: ",".join(f"{k}={v}" for k, v in d.items()))
@pytest.mark.parametrize("launch", [dict(persistent=True), dict(persistent=False), dict(persistent=False, hash_slots=32)],
                         ids=["persistent", "plain", "tiny hash"])
@pytest.mark.parametrize("nq", [2, 200, 500, 700, 1400])
def test_default_launch_by_number_of_queries(sz, collection, kw, launch, nq):
    queries, ix = collection
    q = queries.slice(0, nq)
    kw = dict(dict(k=10, cut=8, heap_factor=0.8), **kw)
    gi, gs, gst = sz.seismic_search(ix, q, stats=True, **launch, **kw)
    ri, rs, rst = sz.seismic_search(ix, q, group=32, persistent=True, stats=True, **dict(kw, cta_warps=8))
    np.testing.assert_array_equal(gs, rs)
    np.testing.assert_array_equal(gi, ri)
    for name in ("lists", "blocks_scored", "blocks_evaluated", "blocks_skipped", "block_docs", "summary_entries"):
        np.testing.assert_array_equal(gst[:, sz.STATS.index(name)], rst[:, sz.STATS.index(name)], err_msg=name)
    if "hash_slots" not in launch:  # a set that forgets scores some documents again
        for name in ("docs", "doc_nnz", "knn_docs", "knn_nnz"):
            np.testing.assert_array_equal(gst[:, sz.STATS.index(name)], rst[:, sz.STATS.index(name)], err_msg=name)


# A server admits three requests per CTA that the GPU holds (9 per SM at least: three CTAs of 8 warps), so that a
# batch's slowest query leaves no CTA idle, or what slot_budget says; results are those of the requests alone.
@pytest.mark.parametrize("cta_warps", [0, 8])
@pytest.mark.parametrize("budget", [0, 100])
def test_server_admission(sz, collection, cta_warps, budget):
    import torch
    queries, ix = collection
    p = sz.search_params(k=10, cut=8, heap_factor=0.8, wave=8, persistent=True, use_knn=True, cta_warps=cta_warps)
    ids, sc = sz.seismic_search(ix, queries, p)
    srv = sz.Server(ix, p, max_batch=128, streams=32, max_query_nnz=100, slot_budget=budget)
    n = 4000
    tickets = []
    for i in range(n):
        a, b = int(queries.indptr[i % queries.n_rows]), int(queries.indptr[i % queries.n_rows + 1])
        tickets.append(srv.submit(queries.terms[a:b], queries.vals[a:b], 10))
    srv.progress()  # admits
    torch.cuda.synchronize()
    done = srv.progress()  # what was admitted has ended
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert done == budget if budget else 9 * sms <= done < n
    while done < n:
        done += srv.progress()
    for i, t in enumerate(tickets):
        gi, gs, _ = srv.result(t, 10)
        np.testing.assert_array_equal(gi, ids[i % queries.n_rows])
        np.testing.assert_array_equal(gs, sc[i % queries.n_rows])
    srv.close()


# The tuner times the launch that the library chooses by itself, and so returns none that is slower.
def test_autotune_reaches_the_default_launch(sz, collection):
    from paper_2509_24815_gb300 import autotune
    queries, ix = collection
    best, table = autotune.autotune(ix, sz.DeviceCSR.from_host(queries.slice(0, 1)), dict(k=10, cut=8, heap_factor=0.8))
    own = [t["ms"] for t in table if t["shape"] == 1 and t["group"] == 1 and t["cta_warps"] == 0]
    assert len(own) == 8
    assert min(t["ms"] for t in table if "ms" in t) <= min(own)
    assert {x: best[x] for x in ("k", "cut", "heap_factor")} == dict(k=10, cut=8, heap_factor=0.8)


# The centroids that clustering takes at a time depend on the vocabulary's bitmap (56 at 500 terms, 51 at 30,522, 48 at
# 45,000, 44 at 65,535): the clusters do not.
def test_clusters_do_not_depend_on_the_vocabulary(sz):
    rng = np.random.default_rng(9)
    docs = _rows(4000, lambda i: rng.integers(0, 500, rng.integers(1, 40)), -2, 9, 500, rng)
    want = None
    for dim in (500, 30522, 45000, 65535):
        ix = sz.seismic_build(synth.CSR(docs.indptr, docs.terms, docs.vals, dim), lambda_=300, beta=150, alpha=0.5, seed=4)
        got = [sz.seismic_export(ix, "cent"), sz.seismic_export(ix, "bdoc")]
        ix.close()
        want = want or got
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a, b)
