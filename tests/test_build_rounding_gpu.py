"""The build's distances against the oracle's tree, bit for bit: dimensions
around the eight lanes and the 16-byte loads of the mapping kernel, exact ties,
duplicates, and coordinates so small or so large that FP32 squares lose bits."""
import numpy as np
import pytest

from oracle.index import build_index
from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gts():
    import paper_2404_00966_gb300 as g
    return g


def same_tree(gts, X, metric, F, h):
    ix = gts.Index.build(X, metric, n_pivots=h, fanout=F, root_pivot=3)
    T = build_index(X, metric, F, h, root_pivot=3)
    for l in range(T["h"] + 1):
        g = ix.tree_level(l)
        assert np.array_equal(g["pos"], T["pos"][l]) and np.array_equal(g["size"], T["size"][l])
        if l < T["h"]:
            assert np.array_equal(g["pivot"], T["pivot"][l])
    ids, tab = ix.table()
    assert np.array_equal(ids, T["perm"])
    assert np.array_equal(tab, T["table"])
    ix.close()


@pytest.mark.parametrize("metric", ["l2", "l1"])
@pytest.mark.parametrize("dim", [8, 9, 16, 31, 32, 33, 100, 128, 300, 1029])
def test_mapped_distances_are_the_rounded_fp64_sums(gts, metric, dim):
    X, _ = small_vectors(3001, dim, 1, seed=400 + dim, dup_frac=0.1)
    same_tree(gts, X, metric, 6, 2)


@pytest.mark.parametrize("metric", ["l2", "l1"])
@pytest.mark.parametrize("scale", [1e-22, 1e-12, 1e12, 1e18])
def test_mapped_distances_at_the_ends_of_the_range(gts, metric, scale):
    X, _ = small_vectors(2003, 40, 1, seed=11)
    same_tree(gts, (X * np.float32(scale)).astype(np.float32), metric, 5, 2)


@pytest.mark.parametrize("metric", ["l2", "l1"])
def test_mapped_distances_with_exact_values(gts, metric):
    """Small integers: sums that FP32 holds exactly, many ties and zeros."""
    X = np.random.default_rng(5).integers(0, 3, size=(2400, 24)).astype(np.float32)
    same_tree(gts, X, metric, 6, 3)
