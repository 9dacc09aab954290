"""Batches of a few queries (default precision) read every row in one pass:
sizes around the four queries of a pass, rows that no 16-byte copy can take,
every k from 1 to beyond the objects, per-query sequence numbers, deletes and
the cache list, and more answers than the first launch has room for -- against
the oracle."""
import numpy as np
import pytest

import oracle
from synth import small_vectors

pytestmark = pytest.mark.gpu
RTOL = 1e-5   # the library's stated distance tolerance


@pytest.fixture(scope="module")
def gts():
    import paper_2404_00966_gb300 as g
    return g


def check(got, want, what):
    off, ids, dist, _ = want
    assert np.array_equal(got.offsets, off), what
    assert np.array_equal(got.ids, ids), what
    assert np.allclose(got.dist, dist, rtol=RTOL, atol=1e-30), what


@pytest.mark.parametrize("metric,dim", [("l2", 2), ("l2", 16), ("l2", 17), ("l2", 128), ("l2", 300), ("l1", 3),
                                        ("l1", 100), ("cos", 3), ("cos", 40)])
@pytest.mark.parametrize("nq", [1, 3, 4, 5, 8, 9])
def test_small_batches(gts, metric, dim, nq):
    X, Q = small_vectors(5003, dim, nq, seed=700 + dim, dup_frac=0.1)
    Q[0] = X[17]
    ix = gts.Index.build(X, metric, fanout=8, root_pivot=3)
    for k in (1, 10, 70, 1024):
        check(ix.knn(Q, k), oracle.knn_query(metric, X, Q, k), f"{metric} {dim} {nq} knn {k}")
    cal = oracle.knn_query(metric, X, Q[:1], 60)
    radii = np.linspace(0.0, 2.0, nq).astype(np.float32) * np.float32(cal[2][-1])
    check(ix.range(Q, radii), oracle.range_query(metric, X, Q, radii), f"{metric} {dim} {nq} range")
    ix.close()


@pytest.mark.parametrize("n", [1, 31, 33, 300])
def test_small_batches_on_few_objects(gts, n):
    X, Q = small_vectors(n, 20, 2, seed=5, kind="uniform")
    ix = gts.Index.build(X, "l2", fanout=4, root_pivot=0)
    check(ix.knn(Q, 40), oracle.knn_query("l2", X, Q, 40), "few objects")
    ix.close()


@pytest.mark.parametrize("metric", ["l2", "l1"])
def test_small_batches_with_updates_and_many_answers(gts, metric):
    X, Q = small_vectors(90_011, 5, 4, seed=8, kind="uniform")
    ix = gts.Index.build(X, metric, fanout=20, root_pivot=0, cache_limit=100_000)
    s0 = ix.info()["seq"]
    extra, _ = small_vectors(200, 5, 1, seed=9, kind="uniform")
    ix.insert(extra)
    dele = np.random.default_rng(3).choice(90_211, 5000, replace=False)
    ix.delete(dele)
    s1 = ix.info()["seq"]
    P = np.concatenate([X, extra])
    ins = np.concatenate([np.full(90_011, -1), s0 + np.arange(200)]).astype(np.int64)
    dl = np.full(P.shape[0], np.iinfo(np.int64).max, np.int64)
    dl[dele] = s0 + 200 + np.arange(5000)
    seq = np.array([s0, s0 + 100, s0 + 200 + 2500, s1], np.int64)
    check(ix.knn(Q, 25, seq=seq), oracle.knn_query(metric, P, Q, 25, ins, dl, seq), "knn at sequence numbers")
    radii = np.full(4, 10.0, np.float32)    # every visible object: past the first launch's room
    check(ix.range(Q, radii, seq=seq), oracle.range_query(metric, P, Q, radii, ins, dl, seq), "all objects")
    ix.close()
