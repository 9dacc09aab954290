"""Batches that keep more pairs than the memory budget holds at once: the tiles and
scans run their blocks in several launches, and the answers are those of the
same call under the default budget, bit for bit."""
import numpy as np
import pytest

from synth import ACGT, LOWER, random_strings, small_vectors

pytestmark = pytest.mark.gpu
GIB = 1 << 30      # 14.5 M pairs; the smallest budget of the default precision's tiles


def arrays(r, nq):
    import torch
    m = r.stats["results"]
    off = torch.zeros(nq + 1, dtype=torch.int64, device="cuda")
    ids = torch.zeros(m, dtype=torch.int64, device="cuda")
    dist = torch.zeros(m, device="cuda")
    r.copy_to(off, ids, dist)
    r.free()
    return off, ids, dist


def same_in_groups(call, per, budget, **kw):
    import torch
    whole = call(*per, result_on_device=True, **kw)
    parts = call(*per, result_on_device=True, memory_budget=budget, **kw)
    assert parts.stats["groups"] > whole.stats["groups"], (parts.stats, whole.stats)
    for a, b in zip(arrays(whole, len(per[1])), arrays(parts, len(per[1]))):
        assert torch.equal(a, b)


@pytest.mark.parametrize("metric,dim,prec,n,nq,budget", [
    ("l2", 24, "fp32", 100_003, 301, GIB), ("cos", 40, "fp32", 100_003, 301, GIB), ("l1", 24, "fp32", 100_003, 301, GIB),
    ("cos", 3, "fp32", 200_003, 120, GIB), ("l1", 24, "bf16", 50_003, 130, 64 << 20)])
def test_range_vectors(metric, dim, prec, n, nq, budget):
    import torch
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(n, dim, nq, seed=dim, kind="uniform")
    ix = gts.Index.build(X, metric, n_pivots=2, fanout=20, root_pivot=0)
    far = 3.2 if metric == "cos" else 1e9                    # every row
    per = (torch.from_numpy(Q).cuda(), torch.full((nq,), far, device="cuda"))
    same_in_groups(ix.range, per, budget, precision=prec)
    ix.close()


@pytest.mark.parametrize("metric,dim,n,nq", [("l2", 3, 200_003, 120), ("l1", 5, 200_003, 120), ("l2", 24, 100_003, 301)])
def test_knn_without_a_bound(metric, dim, n, nq):
    """More neighbours than pivots and no probe: every pair is kept."""
    import torch
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(n, dim, nq, seed=dim, kind="uniform")
    ix = gts.Index.build(X, metric, n_pivots=2, fanout=20, root_pivot=0)
    ix.set_tuning(probe_rows=0)
    per = (torch.from_numpy(Q).cuda(), torch.full((nq,), 1024, dtype=torch.int32, device="cuda"))
    same_in_groups(ix.knn, per, GIB)
    ix.close()


@pytest.mark.parametrize("lo,hi,alpha,n,nq", [(3, 30, LOWER, 100_003, 201),     # filter and distance in one tile
                                              (34, 44, ACGT, 100_003, 201),     # 3-gram filter, integer units
                                              (34, 44, ACGT, 100_003, 450)])    # and tensor cores
def test_range_strings(lo, hi, alpha, n, nq):
    import torch
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(hi)
    S, Q = random_strings(n, lo, hi, alpha, rng), random_strings(nq, lo, hi, alpha, rng)
    ix = gts.Index.build(S, "edit", n_pivots=2, fanout=20, root_pivot=0)
    dev = (torch.from_numpy(Q.data).cuda(), torch.from_numpy(Q.offsets).cuda())
    same_in_groups(ix.range, (dev, torch.full((nq,), 60.0, device="cuda")), GIB)
    ix.close()


def test_a_few_queries_over_more_rows_than_the_budget_takes():
    import torch
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(2_200_003, 2, 8, seed=2, kind="uniform")
    ix = gts.Index.build(X, "l2", n_pivots=2, fanout=20, root_pivot=0)
    per = (torch.from_numpy(Q).cuda(), torch.full((8,), 1e9, device="cuda"))
    one_pass = ix.range(*per, result_on_device=True)
    descent = ix.range(*per, result_on_device=True, memory_budget=GIB)
    assert one_pass.stats["frontier"] == 0 and descent.stats["frontier"] > 0
    for a, b in zip(arrays(one_pass, 8), arrays(descent, 8)):
        assert torch.equal(a, b)
    ix.close()
