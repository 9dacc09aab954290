"""kNN on the tensor-core tiles whose second phase may run with one bf16 product
and its wider bound, against the oracle: every width's tile, ragged rows and
queries, the angle, clustered data (gathered chunks), data far from the origin
(where the bound is too wide and three products stay), deletes."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric,dim,kind,shift", [
    ("l2", 40, "uniform", 0), ("l2", 128, "uniform", 0), ("l2", 190, "uniform", 0), ("l2", 250, "uniform", 0),
    ("l2", 300, "uniform", 0), ("l2", 381, "uniform", 0), ("l2", 440, "uniform", 0), ("cos", 300, "gauss", 0),
    ("l2", 64, "gauss", 0), ("l2", 64, "uniform", 30)])
def test_second_phase(metric, dim, kind, shift):
    import paper_2404_00966_gb300 as gts
    n, nq = 60_013, 301
    X, Q = small_vectors(n, dim, nq, seed=900 + dim, kind=kind, dup_frac=0.05)
    X, Q = X + np.float32(shift), Q + np.float32(shift)
    Q[0] = X[17]
    ix = gts.Index.build(X, metric, n_pivots=4, fanout=12, root_pivot=3)   # 1,728 node blocks
    k = np.resize(np.array([1, 10, 32], np.int32), nq)
    dl = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        r = ix.knn(Q, k, precision="bf16")
        off, ids, dist, _ = oracle.knn_query(metric, X, Q, k, np.full(n, -1, np.int64), dl,
                                             np.full(nq, ix.info()["seq"], np.int64))
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-6)
        s0 = ix.info()["seq"]
        dele = np.random.default_rng(dim).choice(n, 3000, replace=False)
        ix.delete(dele)
        dl[dele] = s0 + np.arange(3000)
    ix.close()
