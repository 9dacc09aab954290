"""Strings over nodes of few and many rows and trees of few nodes: one tile for
filter and distance or the 3-gram tile and the DP, whole and partly filled
blocks, an item's queries in one or several parts; against the oracle, with
deletes."""
import numpy as np
import pytest

import oracle
from synth import ACGT, LOWER, mutate, random_strings, strings_from_list

pytestmark = pytest.mark.gpu


# rows a node: 8, 15, 29 (one group of 32 rows), 48 (two), 75 and 120 (four), 1,500 (20 nodes)
@pytest.mark.parametrize("F,h", [(8, 5), (20, 4), (32, 3), (25, 3), (20, 3), (50, 2), (20, 2)])
@pytest.mark.parametrize("lo,hi,alpha", [(4, 16, LOWER), (24, 32, ACGT), (30, 40, ACGT)])
def test_string_tiles_by_node_rows(F, h, lo, hi, alpha):
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(F + hi)
    n, nq = 30_000, 260
    base = random_strings(900, lo, hi, alpha, rng)
    S = strings_from_list([mutate(base.get(i % 900), int(rng.integers(0, 4)), alpha, rng)[:hi] for i in range(n)])
    Q = strings_from_list([mutate(base.get(i % 900), 2, alpha, rng)[:hi] for i in range(nq)])
    ix = gts.Index.build(S, "edit", n_pivots=h, fanout=F, root_pivot=0)
    some = np.arange(0, nq, 13)
    part = Q.take(some)
    radii = np.resize(np.array([1, 3, 2.5, 5], np.float32), nq)
    k = np.resize(np.array([1, 12, 4], np.int32), nq)
    dele = np.full(n, np.iinfo(np.int64).max, np.int64)
    for step in range(2):
        seq = (np.full(n, -1, np.int64), dele, np.full(len(some), 1, np.int64))
        koff, kids, kdist, _ = oracle.knn_query("edit", S, part, k[some], *seq)
        roff, rids, rdist, _ = oracle.range_query("edit", S, part, radii[some], *seq)
        for prec in ("bf16", "fp32"):
            for r, off, ids, dist in ((ix.knn(Q, k, precision=prec), koff, kids, kdist),
                                      (ix.range(Q, radii, precision=prec), roff, rids, rdist)):
                for j, i in enumerate(some):
                    a, b = r.offsets[i], r.offsets[i + 1]
                    assert np.array_equal(r.ids[a:b], ids[off[j]:off[j + 1]])
                    assert np.array_equal(r.dist[a:b], dist[off[j]:off[j + 1]].astype(np.float32))
        gone = np.unique(kids[::5])
        ix.delete(gone)
        dele[gone] = 0
    ix.close()
