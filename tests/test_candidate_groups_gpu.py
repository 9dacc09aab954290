"""Edit-distance kNN whose candidates exceed the memory budget, so that they are
written and verified in groups: a group's answers lower the thresholds (a
query's entries go over several groups), and the groups after it still write
every candidate that was counted for them.  Against the oracle."""
import numpy as np
import pytest

import oracle
from synth import mutate, random_strings, strings_from_list

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pivots,lo,hi", [(2, 1, 60), (3, 30, 100)])   # nodes of 5,000 rows; of 250
def test_thresholds_lowered_between_candidate_groups(pivots, lo, hi):
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(40 + hi)
    alpha = np.frombuffer(b"abcdefghijklmnopqrstuvwxyz", np.uint8)
    n, nq, k = 100_000, 6, 5
    base = random_strings(40, lo, hi, alpha, rng)
    rows = random_strings(n, lo, hi, alpha, rng)
    rows = [rows.get(i) for i in range(n)]
    for i in range(0, n, 250):            # ten close relatives of each query, among rows of every length
        rows[i] = mutate(base.get((i // 250) % 40), int(rng.integers(0, 4)), alpha, rng)
    S = strings_from_list(rows)
    Q = strings_from_list([mutate(base.get(i), 2, alpha, rng) for i in range(nq)])
    ix = gts.Index.build(S, "edit", n_pivots=pivots, fanout=20, root_pivot=0)
    off, ids, dist, _ = oracle.knn_query("edit", S, Q, k)
    # 6 MiB: groups of at most 85,000 candidates, each enough for the count per distance
    r = ix.knn(Q, k, memory_budget=6 << 20)
    assert r.stats["candidates"] > 3 * 85_000       # (several groups)
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.array_equal(r.dist, dist.astype(np.float32))
    ix.close()
