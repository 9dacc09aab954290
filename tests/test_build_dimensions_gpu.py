"""The build's distances in many dimensions (long sums, whose error bound must stay
narrow) and for row counts off the blocks of 32 rows, against the oracle's
tree, bit for bit."""
import numpy as np
import pytest

from oracle.index import build_index
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric", ["l2", "l1"])
@pytest.mark.parametrize("n,dim", [(1, 24), (31, 24), (33, 17), (1000, 12), (700, 3072), (701, 3075), (400, 8192)])
def test_mapped_distances_of_long_rows_and_ragged_blocks(metric, n, dim):
    import paper_2404_00966_gb300 as gts
    X, _ = small_vectors(n, dim, 1, seed=dim + n, dup_frac=0.05)
    X[n // 2:, 1] *= np.float32(1e5)       # one coordinate far above the others
    ix = gts.Index.build(X, metric, n_pivots=2, fanout=5, root_pivot=0)
    want = build_index(X, metric, 5, 2, root_pivot=0)
    ids, table = ix.table()
    assert np.array_equal(ids, want["perm"]) and np.array_equal(table, want["table"])
    ix.close()
