"""A file whose level offsets are not the tree's (F^l nodes on level l) is refused
before anything is indexed by them."""
import numpy as np
import pytest

from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,by", [(0, 1), (1, -1), (2, 1 << 20), (3, 1), (3, -(1 << 40))])
def test_changed_level_offsets_are_refused(tmp_path, level, by):
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(900, 24, 5, seed=3)
    ix = gts.Index.build(X, "l2", n_pivots=2, fanout=7, root_pivot=0)
    path = tmp_path / "a.gts"
    ix.save(str(path))
    want = ix.knn(Q, 3)
    ix.close()
    off = np.array([0, 1, 8, 57], np.int64)
    data = path.read_bytes()
    assert data.count(off.tobytes()) == 1
    bad = off.copy()
    bad[level] += by
    broken = tmp_path / "b.gts"
    broken.write_bytes(data.replace(off.tobytes(), bad.tobytes()))
    with pytest.raises(gts.GTSError, match="levels"):
        gts.Index.load(str(broken))
    ix = gts.Index.load(str(path))
    assert np.array_equal(ix.knn(Q, 3).ids, want.ids)
    ix.close()
