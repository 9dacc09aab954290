"""Pivot distances of vectors of up to 16 dimensions (a thread per entry) and
of 17 (a warp per entry) against the oracle, with deletes between the batches."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("metric,dim", [("l2", 1), ("l1", 1), ("cos", 2), ("l2", 4), ("l1", 7), ("l2", 15), ("cos", 16),
                                        ("l1", 16), ("l2", 17)])
def test_low_dimensional_pivots(metric, dim, prec):
    import paper_2404_00966_gb300 as gts
    n = 6011
    X, Q = small_vectors(n, dim, 301, seed=700 + dim, kind="uniform", dup_frac=0.1)
    ix = gts.Index.build(X, metric, n_pivots=3, fanout=5, root_pivot=2)
    dl = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        now = np.full(301, ix.info()["seq"], np.int64)
        ins = np.full(n, -1, np.int64)
        kw = (ins, dl, now)
        near = oracle.knn_query(metric, X, Q, 9, *kw)
        radii = near[2][near[0][1:] - 1].astype(np.float32)
        for got, want in ((ix.knn(Q, 9, precision=prec), near),
                          (ix.range(Q, radii, precision=prec), oracle.range_query(metric, X, Q, radii, *kw))):
            assert np.array_equal(got.offsets, want[0]) and np.array_equal(got.ids, want[1])
            assert np.allclose(got.dist, want[2], rtol=1e-5, atol=1e-6)
        s0 = ix.info()["seq"]
        dele = np.random.default_rng(dim).choice(n, 500, replace=False)
        ix.delete(dele)
        dl[dele] = s0 + np.arange(500)
    ix.close()
