"""The dense last level with few parents or few queries, whose blocks take part of a
parent's nodes and of the queries: against the oracle, at the largest and at
odd fanouts, with deletes."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,F,h,nq", [(5003, 64, 2, 601), (9001, 37, 2, 300), (4001, 7, 3, 1030), (3001, 64, 2, 70),
                                      (20011, 20, 2, 2600)])
@pytest.mark.parametrize("metric", ["l2", "cos"])
def test_parts_of_a_parent(metric, n, F, h, nq):
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(n, 40, nq, seed=F + nq, kind="uniform", dup_frac=0.05)
    ix = gts.Index.build(X, metric, n_pivots=h, fanout=F, root_pivot=1)
    off, ids, dist, _ = oracle.knn_query(metric, X, Q, 5)
    r = ix.knn(Q, 5, precision="bf16")
    assert r.stats["dense_last"] == 1
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    radii = dist.reshape(nq, 5)[:, 3].astype(np.float32)
    gone = ids[::11][:60]
    ix.delete(gone)
    dele = np.full(n, np.iinfo(np.int64).max, np.int64)
    dele[gone] = 0
    off, ids, dist, _ = oracle.range_query(metric, X, Q, radii, np.full(n, -1, np.int64), dele, np.full(nq, 1, np.int64))
    r = ix.range(Q, radii, precision="bf16")
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-30)
    ix.close()
