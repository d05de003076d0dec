"""Sizes at which the kernels' tiles, queues and splits end: each against an
exact reference computed here."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _int_rows(n, dim, lo, hi, vlo, vhi, seed):
    """n sparse rows of small whole values: fp32 sums of products are exact, and ties are common."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(lo, hi + 1, n)
    indptr = np.zeros(n + 1, dtype=np.uint64)
    np.cumsum(lens, out=indptr[1:])
    terms = np.concatenate([np.sort(rng.choice(dim, m, replace=False)) for m in lens]) if n else np.empty(0)
    vals = rng.integers(vlo, vhi + 1, int(indptr[-1]))
    vals[vals == 0] = 1
    return synth.CSR(indptr, terms.astype(np.uint16), vals.astype(np.float32), dim)


# one document tile holds 16,384 documents; 3 CTAs per SM decide the splits; k <= 256 has the small sort area
@pytest.mark.parametrize("n_docs", [1000, 16384, 16385, 40001])
@pytest.mark.parametrize("nq,k", [(1, 10), (3, 257), (40, 1024), (600, 256), (600, 1)])
def test_exact_search_tiles_and_splits(sz, n_docs, nq, k):
    dim = 97
    docs = _int_rows(n_docs, dim, 1, 6, -2, 5, 3)
    queries = _int_rows(nq, dim, 0, 40, -2, 3, 4)
    ix = sz.seismic_build(docs, lambda_=20, beta=4, alpha=0.5, seed=1, keep_full_lists=True)
    ids, sc = sz.seismic_search_exact(ix, queries, k)
    ix.close()
    score = queries.to_dense() @ docs.to_dense().T
    order = np.argsort(-score, axis=1, kind="stable")[:, :k]  # score descending, id ascending
    m = order.shape[1]
    np.testing.assert_array_equal(ids[:, :m], order.astype(np.uint32))
    np.testing.assert_array_equal(sc[:, :m], np.take_along_axis(score, order, 1).astype(np.float32))
    assert (ids[:, m:] == sz.NONE_ID).all() and np.isneginf(sc[:, m:]).all()


def _bf16(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).bfloat16().float().numpy().astype(np.float64)


# 32 rows per CTA; gradients off a 16-byte boundary are added one by one.  Bar: fp32 sums of up to 5000 products
# (5000 * 2^-24 = 3e-4) and the bf16 roundings that fall the other way (2^-9 each, few) stay below 1e-2 in norm.
@pytest.mark.parametrize("n", [1, 31, 33, 5000])
@pytest.mark.parametrize("offset", [0, 1])
def test_mlp_gradient_row_edges(sz, n, offset):
    import torch
    from oracle import mlp
    rng = np.random.default_rng(n)
    w = (mlp.init(3) * 0.5).astype(np.float32)
    feat = rng.random((n, 64)).astype(np.float32) * 4
    tgt = rng.random((n, 2)).astype(np.float32)
    buf = [torch.zeros(mlp.N_PARAMS + 4, device="cuda")[offset:offset + mlp.N_PARAMS] for _ in range(4)]
    buf[0].copy_(torch.from_numpy(w))
    loss = torch.zeros(1, device="cuda")
    sz.seismic_mlp_train_step(buf[0], buf[1], buf[2], buf[3], torch.from_numpy(feat).cuda(),
                              torch.from_numpy(tgt).cuda(), 0.0, 1, loss)
    torch.cuda.synchronize()
    p = mlp.unpack(w)
    a0 = _bf16(feat)
    z1 = a0 @ p["W1"].T + p["b1"]
    a1 = _bf16(np.maximum(z1, 0))
    z2 = a1 @ p["W2"].T + p["b2"]
    a2 = _bf16(np.maximum(z2, 0))
    s = mlp.sigmoid(a2 @ p["W3"].T + p["b3"])
    e = s - tgt
    do = 2 * e * s * (1 - s) / n
    d2 = (do @ p["W3"]) * (z2 > 0)
    d1 = (d2 @ p["W2"]) * (z1 > 0)
    ref = mlp.pack(dict(W1=d1.T @ a0, b1=d1.sum(0), W2=d2.T @ a1, b2=d2.sum(0), W3=do.T @ a2, b3=do.sum(0)))
    got = buf[1].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-2 * np.linalg.norm(ref)
    assert abs(loss.item() - (e * e).sum() / n) <= 1e-3 * loss.item()
    np.testing.assert_array_equal(buf[0].cpu().numpy(), w)  # learning rate 0


@pytest.fixture(scope="module", params=[False, True], ids=["fp32", "fp16"])
def dense_hits(sz, request):
    """Whole-valued rows and queries over few terms, so that a row's terms are mostly hits (the candidate queues
    fill), with rows of 1..40 entries, of 300..500, beyond a queue's 2048 positions, and copies of queries."""
    dim = 4000
    short, mid = _int_rows(2500, 300, 1, 40, -1, 4, 11), _int_rows(300, 600, 300, 500, -1, 4, 12)
    long, queries = _int_rows(7, dim, 2049, 2600, 1, 4, 13), _int_rows(330, 520, 1, 400, 1, 3, 14)
    parts = [short, mid, long, queries.slice(0, 60)]
    indptr = np.concatenate([[0]] + [np.diff(p.indptr.astype(np.int64)) for p in parts]).cumsum().astype(np.uint64)
    docs = synth.CSR(indptr, np.concatenate([p.terms for p in parts]), np.concatenate([p.vals for p in parts]), dim)
    queries = synth.CSR(queries.indptr, queries.terms, queries.vals, dim)
    ix = sz.seismic_build(docs, lambda_=400, beta=60, alpha=0.6, quantize_u8=False, seed=2, values_fp16=request.param)
    yield docs, queries, ix
    ix.close()


# Lane groups score one row at a time and one wave at a time; sums of whole values are exact in any order, so the
# documents, the scores and the work counted have to be the same.
@pytest.mark.parametrize("kw", [dict(wave=1), dict(wave=1, heap_factor=1.3), dict(wave=3, heap_factor=1.0),
                                dict(wave=2, hf_mode=1, heap_factor=0.8), dict(wave=64), dict(exhaustive=True)],
                         ids=lambda d: ",".join(f"{k}={v}" for k, v in d.items()))
@pytest.mark.parametrize("launch", [dict(persistent=True), dict(persistent=True, cta_warps=4), dict(persistent=False),
                                    dict(persistent=False, hash_slots=16)],
                         ids=["persistent", "4 warps", "plain", "tiny hash"])
@pytest.mark.parametrize("nq,k", [(1, 3), (200, 10), (330, 60)])
def test_group_1_equals_lane_groups(sz, dense_hits, kw, launch, nq, k):
    _, queries, ix = dense_hits
    q = queries.slice(0, nq)
    kw = dict(dict(cut=9, heap_factor=0.9), k=k, **kw) if "heap_factor" not in kw else dict(cut=9, k=k, **kw)
    gi, gs, gst = sz.seismic_search(ix, q, group=1, stats=True, **launch, **kw)
    ri, rs, rst = sz.seismic_search(ix, q, group=32, cta_warps=8, persistent=True, stats=True, **kw)
    np.testing.assert_array_equal(gs, rs)
    np.testing.assert_array_equal(gi, ri)
    for name in ("lists", "blocks_scored", "blocks_evaluated", "blocks_skipped", "block_docs", "summary_entries"):
        np.testing.assert_array_equal(gst[:, sz.STATS.index(name)], rst[:, sz.STATS.index(name)], err_msg=name)
    if "hash_slots" not in launch:  # a set that forgets scores some documents again
        for name in ("docs", "doc_nnz"):
            np.testing.assert_array_equal(gst[:, sz.STATS.index(name)], rst[:, sz.STATS.index(name)], err_msg=name)


def test_group_1_graph_stages_equal_lane_groups(sz, dense_hits):
    docs, queries, ix = dense_hits
    rng = np.random.default_rng(5)
    sz.seismic_set_knn(ix, rng.integers(0, docs.n_rows, (docs.n_rows, 7)))
    for launch in (dict(persistent=True), dict(persistent=False, hash_slots=16)):
        for nq in (3, 330):
            got = sz.seismic_search(ix, queries.slice(0, nq), k=50, cut=2, heap_factor=1.0, use_knn=True, **launch)
            ref = sz.seismic_search(ix, queries.slice(0, nq), k=50, cut=2, heap_factor=1.0, use_knn=True, group=16,
                                    persistent=True)
            np.testing.assert_array_equal(got[1], ref[1])
            np.testing.assert_array_equal(got[0], ref[0])


# Masses spread over more than 53 bits are added one after the other, others as integers: both give the prefix of
# sequential fp64 sums.  Codes are quantised in fp64 from the kept values.
@pytest.mark.parametrize("spread", [0, 12, 40])
@pytest.mark.parametrize("alpha", [0.05, 0.4, 1.0])
def test_summary_masses_and_codes(sz, spread, alpha):
    rng = np.random.default_rng(spread)
    docs = _int_rows(700, 3000, 1, 300, 1, 3, 21)
    vals = (rng.random(docs.nnz) + 0.5) * np.exp2(rng.integers(-spread, 1, docs.nnz)) * rng.choice([1, 1, 1, -1], docs.nnz)
    docs = synth.CSR(docs.indptr, docs.terms, vals.astype(np.float32), docs.dim)
    ix = sz.seismic_build(docs, lambda_=60, beta=7, alpha=alpha, quantize_u8=True, seed=1, keep_block_summaries=True)
    x = {n: sz.seismic_export(ix, n) for n in ("bdoc_ptr", "bdoc", "sum_ptr", "sum_term", "sum_val", "sum_code")}
    ix.close()
    dense = docs.to_dense()
    blocks = rng.choice(len(x["bdoc_ptr"]) - 1, 400, replace=False)
    for g in blocks:
        phi = dense[x["bdoc"][x["bdoc_ptr"][g]:x["bdoc_ptr"][g + 1]]].max(axis=0)
        order = np.lexsort((np.arange(docs.dim), -np.abs(phi)))
        order = order[phi[order] != 0]
        mass = np.cumsum(np.abs(phi[order]))
        keep = order[:int(np.argmax(mass >= alpha * mass[-1])) + 1] if len(order) else order
        a, b = int(x["sum_ptr"][g]), int(x["sum_ptr"][g + 1])
        keep = np.sort(keep)
        np.testing.assert_array_equal(x["sum_term"][a:b], keep)
        np.testing.assert_array_equal(x["sum_val"][a:b], phi[keep].astype(np.float32))
        if len(keep):
            m, size = phi[keep].min(), float(np.float32((phi[keep].max() - phi[keep].min()) / 256.0))
            code = np.clip(np.floor((phi[keep] - m) / size), 0, 255) if size > 0 else np.zeros(len(keep))
            np.testing.assert_array_equal(x["sum_code"][a:b], code.astype(np.uint8))


# A shared-memory budget that holds for the query alone: long queries leave group 1 for lane groups, past 200 KB
# they are refused, whatever the seen set.
def test_long_queries_and_the_shared_memory_limit(sz):
    dim = 40000
    docs = _int_rows(500, dim, 1000, 3000, 1, 3, 31)
    q = _int_rows(3, dim, 6000, 9000, 1, 2, 32)
    ix = sz.seismic_build(docs, lambda_=50, beta=5, alpha=0.5, quantize_u8=False, seed=1)
    for kw in (dict(), dict(persistent=True), dict(cta_warps=16), dict(hash_slots=64)):
        got = sz.seismic_search(ix, q, k=5, cut=40, heap_factor=1.0, **kw)
        ref = sz.seismic_search(ix, q, k=5, cut=40, heap_factor=1.0, group=8, persistent=True, cta_warps=kw.get("cta_warps", 8))
        np.testing.assert_array_equal(got[1], ref[1])
        np.testing.assert_array_equal(got[0], ref[0])
    with pytest.raises(sz.SeismicError) as e:
        sz.seismic_search(ix, _int_rows(2, dim, 14000, 15000, 1, 2, 33), k=5, cut=40)
    assert e.value.code == sz.EBUDGET
    ix.close()
