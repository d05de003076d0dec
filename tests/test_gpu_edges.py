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
