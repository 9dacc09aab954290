"""Large range answer sets (at least 2^19 answers) are grouped by query and
piece of the id range and ranked within these runs of up to 256; longer runs
(ids bunched around a query) take the device-wide sort.  Both against the
oracle, with empty queries, heavy queries, cache-list answers and deletes."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu
MEAN, LONGEST = 48, 256


@pytest.fixture(scope="module")
def gts():
    import paper_2404_00966_gb300 as g
    return g


def longest_run(off, ids, n):
    most = 0
    for q in range(off.size - 1):
        a = ids[off[q]:off[q + 1]].astype(object)
        pieces = a.size // MEAN + 1
        mul = (pieces << 32) // n
        if a.size:
            most = max(most, int(np.bincount(np.array([int(i) * mul >> 32 for i in a])).max()))
    return most


def same(r, want):
    off, ids, dist, _ = want
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.allclose(r.dist, dist, rtol=1e-5, atol=1e-30)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("metric,dim", [("l2", 2), ("l1", 3), ("l2", 4)])
def test_range_answer_runs(gts, metric, dim, prec):
    X, Q = small_vectors(20_011, dim, 600, seed=500 + dim, kind="uniform")
    ix = gts.Index.build(X, metric, fanout=8, root_pivot=1, cache_limit=100_000)
    s0 = ix.info()["seq"]
    extra, _ = small_vectors(300, dim, 1, seed=501, kind="uniform")
    ix.insert(extra)
    dele = np.random.default_rng(7).choice(20_311, 400, replace=False)
    ix.delete(dele)
    P = np.concatenate([X, extra])
    ins = np.concatenate([np.full(20_011, -1), s0 + np.arange(300)]).astype(np.int64)
    dl = np.full(P.shape[0], np.iinfo(np.int64).max, np.int64)
    dl[dele] = s0 + 300 + np.arange(400)
    near = np.sort(oracle.distances_to(metric, X, Q[0]))
    radii = np.resize(near[[1900, 2000, 2100, 600]].astype(np.float32), 600)
    radii[::50] = 0.0                       # queries of no answer
    radii[7] = np.float32(near[9000])       # a heavy query
    want = oracle.range_query(metric, P, Q, radii, ins, dl, np.full(600, ix.info()["seq"], np.int64))
    assert want[0][-1] >= 1 << 19 and longest_run(want[0], want[1], 20_311) <= LONGEST
    same(ix.range(Q, radii, precision=prec), want)
    ix.close()


@pytest.mark.parametrize("share,lo,hi", [(0.3, 128, LONGEST), (1.0, LONGEST, 1 << 30)])
def test_range_answers_with_bunched_ids(gts, share, lo, hi):
    """About 430 answers a query of points on a line; `share` of them sit in
    the line's order, so that a query's answers among them have neighbouring
    ids: runs of 129 to 256 answers, and runs no warp sorts."""
    n, nq = 20_011, 1300
    X, Q = small_vectors(n, 1, nq, seed=502, kind="uniform")
    near = np.sort(oracle.distances_to("l2", X, Q[0]))
    radii = np.full(nq, near[440], np.float32)
    m = int(share * n)
    X[:m] = np.sort(X[:m], axis=0)
    want = oracle.range_query("l2", X, Q, radii)
    assert want[0][-1] >= 1 << 19
    assert lo < longest_run(want[0], want[1], n) <= hi
    ix = gts.Index.build(X, "l2", fanout=8, root_pivot=1)
    same(ix.range(Q, radii, precision="bf16"), want)
    ix.close()
