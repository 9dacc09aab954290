"""A batch that kept most of the rows must not size the outputs of later batches
beyond the memory budget (every route that remembers its output size)."""
import numpy as np
import pytest

from synth import small_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric,dim", [("l2", 24), ("l1", 24), ("l2", 3)])
def test_a_wide_batch_then_a_larger_narrow_one(metric, dim):
    import torch
    import paper_2404_00966_gb300 as gts
    n, nq = 100_000, 400_000
    X, _ = small_vectors(n, dim, 1, seed=dim, kind="uniform")
    X[:, 0] = np.arange(n, dtype=np.float32) * np.float32(0.25)      # no two rows alike
    Xd = torch.from_numpy(X).cuda()
    ix = gts.Index.build(Xd, metric, n_pivots=2, fanout=20, root_pivot=0)
    wide = ix.range(Xd[:300].contiguous(), torch.full((300,), 1e9, device="cuda"), result_on_device=True,
                    memory_budget=4 << 30)
    assert wide.stats["results"] == 300 * n          # 10^5 pairs a query
    wide.free()
    # twice that per query, for 400,000 queries, would be 8 * 10^10 pairs
    Q = Xd.repeat(nq // n, 1).contiguous()
    r = ix.range(Q, torch.zeros(nq, device="cuda"), memory_budget=4 << 30)
    assert np.array_equal(r.offsets, np.arange(nq + 1)) and np.array_equal(r.ids, np.tile(np.arange(n), nq // n))
    ix.close()
