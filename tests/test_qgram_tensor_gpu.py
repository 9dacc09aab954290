"""The 3-gram bound on the tensor cores (large, well-filled batches of strings)
against the same queries in batches too small for it, and a few against the
oracle: ordinary reads, repeats (3-gram counts far above the cap), a byte
alphabet; whole and fractional radii, none, and one that keeps every pair; kNN;
deletes; row and query counts off the 128-row and 256-query tiles."""
import numpy as np
import pytest

import oracle
from synth import ACGT, mutate, random_strings, strings_from_list

pytestmark = pytest.mark.gpu
N, NQ = 70_011, 521   # 36 M pairs at once, 3.6 M in batches of 53


def reads(kind, count, rng, base):
    out = []
    for i in range(count):
        if kind == "repeats" and i % 3 == 0:
            unit = bytes(rng.choice(ACGT, int(rng.integers(1, 4))))
            s = mutate((unit * 300)[:int(rng.integers(40, 290))], int(rng.integers(0, 4)), ACGT, rng)
        else:
            s = mutate(base.get(int(rng.integers(0, 900))), int(rng.integers(0, 9)), ACGT, rng)
        out.append(s)
    return out


@pytest.mark.parametrize("kind", ["reads", "repeats", "bytes"])
def test_tensor_filter_matches_small_batches(kind):
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(81)
    if kind == "bytes":
        alpha = np.arange(33, 123, dtype=np.uint8)
        base = random_strings(900, 33, 60, alpha, rng)
    else:
        base = random_strings(900, 60, 108, ACGT, rng)
    S = strings_from_list(reads(kind, N, rng, base))
    queries = reads(kind, NQ, rng, base)
    ix = gts.Index.build(S, "edit", n_pivots=2, fanout=20, root_pivot=0)
    radii = np.resize(np.array([8, 9, 6.5, 8, 12, 7, 8, 0], np.float32), NQ)
    radii[100] = 400.0
    k = np.resize(np.array([1, 5, 17], np.int32), NQ)
    for step in range(2):
        Q = strings_from_list(queries)
        big_r = ix.range(Q, radii, precision="bf16")
        big_k = ix.knn(Q, k, precision="bf16")
        for a in range(0, NQ, 53):
            b = min(a + 53, NQ)
            part = strings_from_list(queries[a:b])
            for big, small in ((big_r, ix.range(part, radii[a:b], precision="fp32")),
                               (big_k, ix.knn(part, k[a:b], precision="fp32"))):
                lo, hi = big.offsets[a], big.offsets[b]
                assert np.array_equal(big.offsets[a:b + 1] - lo, small.offsets)
                assert np.array_equal(big.ids[lo:hi], small.ids) and np.array_equal(big.dist[lo:hi], small.dist)
        if step == 0:
            some = [0, 1, 300]
            off, ids, dist, _ = oracle.range_query("edit", S, strings_from_list([queries[i] for i in some]), radii[some])
            for j, i in enumerate(some):
                assert np.array_equal(big_r.ids[big_r.offsets[i]:big_r.offsets[i + 1]], ids[off[j]:off[j + 1]])
            ix.delete(rng.choice(N, 5000, replace=False))
    ix.close()
