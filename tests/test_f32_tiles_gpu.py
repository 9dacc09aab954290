"""The FP32 node tiles (the default precision on batches) against the oracle:
edges of the 128-row blocks, of the 32 / 64 / 128-query chunks and of the
32-coordinate slices, rows that no 16-byte copy can take, and deletes."""
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
    assert np.allclose(got.dist, dist, rtol=RTOL, atol=0), what


@pytest.mark.parametrize("metric,dim", [("l2", 17), ("l2", 32), ("l2", 33), ("l2", 100), ("l2", 128), ("l2", 300),
                                        ("l1", 20), ("l1", 100), ("cos", 24)])
@pytest.mark.parametrize("nq", [33, 130, 300])
def test_f32_tiles_match_the_oracle(gts, metric, dim, nq):
    n = {33: 400011, 130: 100011, 300: 50011}[nq]   # enough (query, row) pairs for the tiles in every case
    X, Q = small_vectors(n, dim, nq, seed=200 + dim, kind="uniform", dup_frac=0.1)
    Q[:3] = X[[5, 9, n - 1]]
    ix = gts.Index.build(X, metric, n_pivots=2, fanout=6, root_pivot=7)   # six nodes of many blocks
    for k in (1, 10, 70):
        r = ix.knn(Q, k)
        assert r.stats["tiles"] > 0
        check(r, oracle.knn_query(metric, X, Q, k), f"{metric} {dim} knn {k}")
    cal = oracle.knn_query(metric, X, Q[:10], 40)
    radii = np.linspace(0.0, 1.2, nq).astype(np.float32) * np.float32(np.mean(cal[2][cal[0][1:] - 1]))
    check(ix.range(Q, radii), oracle.range_query(metric, X, Q, radii), f"{metric} {dim} range")
    ix.close()


def test_f32_tiles_unaligned_queries_and_deletes(gts):
    """Device queries that start 4 bytes past a 16-byte boundary take the
    4-byte copies; deleted rows are skipped at the query's sequence number."""
    import torch
    X, Q = small_vectors(80011, 64, 200, seed=9, kind="uniform")
    buf = torch.zeros(200 * 64 + 1, device="cuda")
    buf[1:] = torch.from_numpy(Q.reshape(-1)).cuda()
    Qd = buf[1:].view(200, 64)
    assert Qd.data_ptr() % 16 == 4
    ix = gts.Index.build(X, "l2", n_pivots=2, fanout=6, root_pivot=0)
    s0 = ix.info()["seq"]
    dele = np.random.default_rng(3).choice(80011, 500, replace=False)
    ix.delete(dele)
    s1 = ix.info()["seq"]
    dl = np.full(80011, np.iinfo(np.int64).max, np.int64)
    dl[dele] = s0 + np.arange(500)
    ins = np.full(80011, -1, np.int64)
    r = ix.knn(Qd, torch.full((200,), 12, dtype=torch.int32, device="cuda"))
    assert r.stats["tiles"] > 0
    check(r, oracle.knn_query("l2", X, Q, 12, ins, dl, np.full(200, s1, np.int64)), "deletes")
    ix.close()


@pytest.mark.parametrize("dim", [40, 128, 300])
def test_range_tiles_over_the_parents_of_small_nodes(gts, dim):
    """Range queries on nodes of a few rows run the tensor-core tiles over the
    level above (masks over the nodes, path distances of fewer levels)."""
    X, Q = small_vectors(9011, dim, 210, seed=600 + dim, dup_frac=0.1)
    Q[:3] = X[[5, 9, 9010]]
    ix = gts.Index.build(X, "l2", n_pivots=3, fanout=7, root_pivot=7)   # 49 nodes of 184 rows, 343 of 26
    cal = oracle.knn_query("l2", X, Q[:10], 200)
    radii = np.linspace(0.0, 1.5, 210).astype(np.float32) * np.float32(np.mean(cal[2][cal[0][1:] - 1]))
    r = ix.range(Q, radii, precision="bf16")
    assert r.stats["tiles"] <= 49 * 2 and r.stats["tiles"] > 0      # blocks of the parents, not of the 343 nodes
    check(r, oracle.range_query("l2", X, Q, radii), f"coarse range {dim}")
    ix.close()
