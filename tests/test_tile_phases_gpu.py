"""kNN on the tensor-core tiles with enough node blocks for two phases (the
second with the thresholds the first one's answers give), against the oracle:
windows and gathered chunks, the angle, k past a phase's candidates, deletes."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric,dim,nq,kind", [("l2", 17, 130, "uniform"), ("l2", 128, 257, "uniform"),
                                                ("l2", 40, 65, "gauss"), ("cos", 70, 130, "uniform"),
                                                ("cos", 300, 64, "uniform")])
def test_two_phases(metric, dim, nq, kind):
    import paper_2404_00966_gb300 as gts
    n = 30_011
    X, Q = small_vectors(n, dim, nq, seed=800 + dim, kind=kind, dup_frac=0.1)
    ix = gts.Index.build(X, metric, n_pivots=4, fanout=12, root_pivot=3)   # 1,728 node blocks
    k = np.resize(np.array([1, 10, 40, 300], np.int32), nq)
    dl = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        r = ix.knn(Q, k, precision="bf16")
        if kind == "uniform":
            assert r.stats["tiles"] >= 1216
        off, ids, dist, _ = oracle.knn_query(metric, X, Q, k, np.full(n, -1, np.int64), dl,
                                             np.full(nq, ix.info()["seq"], np.int64))
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-6)
        s0 = ix.info()["seq"]
        dele = np.random.default_rng(dim).choice(n, 2000, replace=False)
        ix.delete(dele)
        dl[dele] = s0 + np.arange(2000)
    ix.close()
