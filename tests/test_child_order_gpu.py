"""Children tested as one range of a node's rising child intervals, and one by
one where the intervals do not rise (a file whose bounds were widened): both
against the oracle, with nodes of fewer rows than children and equal distances."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gts():
    import paper_2404_00966_gb300 as g
    return g


def same(got, want):
    off, ids, dist, _ = want
    assert np.array_equal(got.offsets, off) and np.array_equal(got.ids, ids)
    assert np.allclose(got.dist, dist, rtol=1e-5, atol=1e-30)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("metric,dim,n,F,h", [("l2", 3, 5003, 20, 2), ("l1", 24, 700, 32, 2), ("l2", 24, 9001, 6, 4),
                                              ("cos", 20, 3001, 64, 1)])
def test_children_in_order_and_not(gts, tmp_path, metric, dim, n, F, h, prec):
    X, Q = small_vectors(n, dim, 65, seed=600 + dim, kind="uniform", dup_frac=0.3)
    Q[0] = X[3]
    ix = gts.Index.build(X, metric, n_pivots=h, fanout=F, root_pivot=1)
    near = oracle.knn_query(metric, X, Q, 20)
    radii = near[2][near[0][1:] - 1].astype(np.float32)
    radii[5::9] = 0.0
    want_r, want_k = oracle.range_query(metric, X, Q, radii), oracle.knn_query(metric, X, Q, 7)
    same(ix.range(Q, radii, precision=prec), want_r)
    same(ix.knn(Q, 7, precision=prec), want_k)
    path = tmp_path / "a.gts"
    ix.save(str(path))
    hi = np.concatenate([ix.tree_level(l)["hi"] for l in range(h + 1)]).astype(np.float32)
    ix.close()
    data = path.read_bytes()
    assert data.count(hi.tobytes()) == 1
    wide = hi.copy()
    wide[1::3] = np.where(wide[1::3] > 0, wide[1::3] * np.float32(3), wide[1::3])   # wider: still every row inside
    path.write_bytes(data.replace(hi.tobytes(), wide.tobytes()))
    ix = gts.Index.load(str(path))
    same(ix.range(Q, radii, precision=prec), want_r)
    same(ix.knn(Q, 7, precision=prec), want_k)
    ix.close()
