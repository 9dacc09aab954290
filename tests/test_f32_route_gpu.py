"""FP32 batches over trees of small nodes: tiles or candidate by candidate, by the
rows of a node and the share of the pairs that the table bound leaves; both
against the oracle, with deletes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def data(kind, n, dim, nq, seed):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        return rng.random((n, dim), dtype=np.float32), rng.random((nq, dim), dtype=np.float32)
    centers = rng.uniform(-1, 1, (64, dim))

    def some(m):
        return (centers[rng.integers(0, 64, m)] + 0.1 * rng.standard_normal((m, dim))).astype(np.float32)
    return some(n), some(nq)


# rows a node 14 (F = 8, five levels) and 7 (n = 30,011)
@pytest.mark.parametrize("metric,kind,n,dim,nq,tiles", [
    ("l1", "uniform", 60_011, 24, 300, True),        # every pair is a candidate: 17 M
    ("l2", "uniform", 60_011, 24, 300, True),
    ("cos", "uniform", 60_011, 20, 300, True),
    ("l1", "gauss", 60_011, 256, 300, False),        # few candidates, wide rows, blocks a ninth full
    ("l1", "uniform", 30_011, 24, 300, False),       # too few rows a node
    ("l2", "uniform", 30_011, 24, 300, False)])
def test_tiles_only_where_the_nodes_fill_them(metric, kind, n, dim, nq, tiles):
    import paper_2404_00966_gb300 as gts
    X, Q = data(kind, n, dim, nq, seed=dim + nq)
    Q[:2] = X[[7, n - 1]]
    ix = gts.Index.build(X, metric, n_pivots=5, fanout=8, root_pivot=3)
    r = ix.knn(Q, 7)
    assert (r.stats["tiles"] > 0) == tiles, r.stats
    off, ids, dist, _ = oracle.knn_query(metric, X, Q, 7)
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-30)
    radii = dist.reshape(nq, 7)[:, 5].astype(np.float32)
    ix.delete(ids[::7][:40])
    dele = np.full(n, np.iinfo(np.int64).max, np.int64)
    dele[ids[::7][:40]] = 0
    r = ix.range(Q, radii)
    off, want, dist, _ = oracle.range_query(metric, X, Q, radii, np.full(n, -1, np.int64), dele, np.full(nq, 1, np.int64))
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, want)
    assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-30)
    ix.close()
