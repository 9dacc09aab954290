"""kNN thresholds from the pivots of a wide level: the gate of the 128 minima
(k up to 128, 512 entries and more), its second pass where most pivots are
deleted, and larger k without it, against the oracle."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("metric,dim", [("l2", 24), ("l1", 20), ("l2", 3)])
def test_thresholds_of_wide_levels(metric, dim, prec):
    import paper_2404_00966_gb300 as gts
    n, nq = 9_001, 41
    X, Q = small_vectors(n, dim, nq, seed=1000 + dim, kind="uniform", dup_frac=0.2)
    ix = gts.Index.build(X, metric, n_pivots=3, fanout=30, root_pivot=0)   # 900 nodes on the last level
    k = np.resize(np.array([1, 32, 33, 100, 128, 129, 500], np.int32), nq)
    dl = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        r = ix.knn(Q, k, precision=prec)
        off, ids, dist, _ = oracle.knn_query(metric, X, Q, k, np.full(n, -1, np.int64), dl,
                                             np.full(nq, ix.info()["seq"], np.int64))
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-6)
        # four fifths of the objects go, the pivots of the last level among them
        s0 = ix.info()["seq"]
        piv = ix.tree_level(2)["pivot"]
        gone = np.random.default_rng(dim).choice(n, 4 * n // 5, replace=False)
        dele = np.unique(np.concatenate([gone, piv[piv >= 0][:800]])) if step == 0 else np.zeros(0, np.int64)
        if dele.size:
            ix.delete(dele)
            dl[dele] = s0 + np.arange(dele.size)
    ix.close()
