"""kNN on few dimensions: the table scan decides the pairs or hands candidates on, by
the candidates that a sample of the entries has; both against the oracle, with
deletes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric,dim,k", [("l2", 16, 1), ("l2", 16, 200), ("l1", 9, 2), ("l1", 9, 300), ("cos", 12, 1),
                                          ("cos", 12, 150), ("l2", 4, 3), ("l2", 5, 3)])
@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_scan_with_few_and_many_candidates(metric, dim, k, prec):
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(dim + k)
    n, nq = 40_009, 900
    centers = rng.uniform(-1, 1, (300, dim))
    X = (centers[rng.integers(0, 300, n)] + 0.05 * rng.standard_normal((n, dim))).astype(np.float32)
    Q = (centers[rng.integers(0, 300, nq)] + 0.05 * rng.standard_normal((nq, dim))).astype(np.float32)
    ix = gts.Index.build(X, metric, n_pivots=4, fanout=8, root_pivot=0)      # 512 nodes of 78 rows
    dele = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        off, ids, dist, _ = oracle.knn_query(metric, X, Q, k, np.full(n, -1, np.int64), dele, np.full(nq, 1, np.int64))
        r = ix.knn(Q, k, precision=prec)
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-6)
        gone = np.unique(ids[::max(1, k)][:300])
        ix.delete(gone)
        dele[gone] = 0
    ix.close()
