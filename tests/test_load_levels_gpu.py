"""Altered index files: level offsets that are not the tree's (F^l nodes on level l)
and string offsets that fall are refused before anything is indexed by them, and
the longest string is taken from the offsets."""
import numpy as np
import pytest

from synth import LOWER, random_strings, small_vectors

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


def test_a_files_word_for_the_longest_string_is_not_taken(tmp_path):
    """kNN counts candidates per distance in a table as wide as the longest string:
    a file that states a shorter one (tree or cache list) answers as before, and
    offsets that fall are refused."""
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(8)
    S, extra = random_strings(20_000, 40, 60, LOWER, rng), random_strings(30, 100, 110, LOWER, rng)
    Q = random_strings(12, 1, 8, LOWER, rng)
    ix = gts.Index.build(S, "edit", n_pivots=1, fanout=20, root_pivot=0)
    ix.insert(extra)
    path = tmp_path / "a.gts"
    ix.save(str(path))
    want = ix.knn(Q, 1024)
    ix.close()
    data = bytearray(path.read_bytes())
    assert np.frombuffer(data[32:36], np.int32)[0] == 60              # the tree's longest string
    data[32:36] = np.int32(3).tobytes()
    cache = np.array([30], np.int64).tobytes() + np.array([110], np.int32).tobytes()
    assert data.count(cache) == 1
    at = data.index(cache) + 8
    data[at:at + 4] = np.int32(2).tobytes()
    short = tmp_path / "b.gts"
    short.write_bytes(data)
    ix = gts.Index.load(str(short))
    got = ix.knn(Q, 1024)
    assert np.array_equal(got.ids, want.ids) and np.array_equal(got.dist, want.dist)
    ix.close()
    off = S.offsets.astype(np.int64)
    data = path.read_bytes()
    # the tree's offsets are in leaf order: find them by their length and their end
    size = np.array([(S.n + 1) * 8], np.int64).tobytes()
    at = data.index(size) + 8
    soff = np.frombuffer(data[at:at + (S.n + 1) * 8], np.int64).copy()
    assert soff[0] == 0 and soff[-1] == off[-1]
    soff[100] = soff[102] + 1
    broken = tmp_path / "c.gts"
    broken.write_bytes(data[:at] + soff.tobytes() + data[at + soff.nbytes:])
    with pytest.raises(gts.GTSError, match="string offsets"):
        gts.Index.load(str(broken))
