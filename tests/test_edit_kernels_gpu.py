"""The edit-distance kernels at the edges of their words and bands: pattern
lengths around 32 / 64 / 128 / 256 / 512 / 1024 characters (one to 32 words
per column) and thresholds around 15 and 31 (the 32- and 64-bit bands),
against the oracle.  Distances are whole numbers: equality."""
import numpy as np
import pytest

import oracle
from synth import ACGT, mutate, random_strings, strings_from_list

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gts():
    import paper_2404_00966_gb300 as g
    return g


def family(lo, hi, n, nq, seed, edits):
    """Strings of length lo .. hi around few seeds, some many edits apart."""
    rng = np.random.default_rng(seed)
    base = random_strings(12, lo, hi, ACGT, rng)
    seeds = [base.get(i) for i in range(12)]

    def some(m):
        out = []
        for _ in range(m):
            s = mutate(seeds[int(rng.integers(0, 12))], int(rng.integers(0, edits + 1)), ACGT, rng)
            out.append(s[:hi])
        return strings_from_list(out)
    return some(n), some(nq)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("lo,hi", [(1, 8), (1, 32), (29, 32), (1, 33), (31, 34), (60, 70), (100, 130), (126, 131), (250, 262), (508, 520),
                                   (1000, 1024)])
def test_edit_bands_and_words(gts, prec, lo, hi):
    n, nq = (700, 48) if hi <= 140 else (260, 24)
    S, Q = family(lo, hi, n, nq, 300 + hi, 44)
    ix = gts.Index.build(S, "edit", n_pivots=2, fanout=5, root_pivot=0)
    radii = np.resize(np.array([0, 1, 7, 14, 15, 16, 30, 31, 32, 45], np.float32), nq)
    off, ids, dist, _ = oracle.range_query("edit", S, Q, radii)
    r = ix.range(Q, radii, precision=prec)
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.array_equal(r.dist, dist.astype(np.float32))
    for k in (1, 9):
        off, ids, dist, _ = oracle.knn_query("edit", S, Q, k)
        r = ix.knn(Q, k, precision=prec)
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.array_equal(r.dist, dist.astype(np.float32))
    ix.close()


def test_edit_bands_saved_and_cached_strings(gts, tmp_path):
    """A loaded index and cache-list strings (their own buffers, any byte alignment)."""
    S, Q = family(90, 128, 500, 40, 7, 20)
    extra, _ = family(90, 128, 61, 1, 8, 20)
    ix = gts.Index.build(S, "edit", n_pivots=2, fanout=5, root_pivot=0)
    ix.insert(extra)
    p = str(tmp_path / "ix.gts")
    ix.save(p)
    jx = gts.Index.load(p)
    both = strings_from_list([S.get(i) for i in range(S.n)] + [extra.get(i) for i in range(extra.n)])
    radii = np.full(40, 12, np.float32)
    off, ids, dist, _ = oracle.range_query("edit", both, Q, radii)
    for index in (ix, jx):
        r = index.range(Q, radii)
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.array_equal(r.dist, dist.astype(np.float32))
    ix.close()
    jx.close()


def test_range_without_the_last_pivot_level(gts):
    """Reads in many small families: the 3-gram filter lets almost nothing
    through, so the rows of the last level are filtered without its pivots
    (fewer pivot distances than entries); deleted rows stay out; radii on both
    sides of the filter's whole-number limit."""
    rng = np.random.default_rng(77)
    base = random_strings(600, 100, 108, ACGT, rng)
    items = [mutate(base.get(i % 600), int(rng.integers(0, 7)), ACGT, rng) for i in range(6007)]
    S = strings_from_list(items)
    Q = strings_from_list([mutate(base.get(int(rng.integers(0, 600))), int(rng.integers(0, 7)), ACGT, rng)
                           for _ in range(201)])
    ix = gts.Index.build(S, "edit", n_pivots=3, fanout=6, root_pivot=0)
    radii = np.resize(np.array([0, 1, 8, 9], np.float32), 201)
    s0 = ix.info()["seq"]
    dele = rng.choice(6007, 300, replace=False)
    for step in range(2):
        r = ix.range(Q, radii, precision="bf16")
        assert r.stats["pivot_dist"] < r.stats["frontier"]
        ins = np.full(6007, -1, np.int64)
        dl = np.full(6007, np.iinfo(np.int64).max, np.int64)
        if step:
            dl[dele] = s0 + np.arange(300)
        off, ids, dist, _ = oracle.range_query("edit", S, Q, radii, ins, dl,
                                               np.full(201, ix.info()["seq"], np.int64))
        assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
        assert np.array_equal(r.dist, dist.astype(np.float32))
        if not step:
            ix.delete(dele)
    ix.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_short_string_tiles(gts, prec):
    """Words: both precisions run the filter and the distance in one tile once
    the batch holds 6 M (entry, row) pairs; deleted rows stay out."""
    rng = np.random.default_rng(9)
    alpha = np.frombuffer(b"abcdefghijklmnopqrstuvwxyz", np.uint8)
    S = random_strings(40_003, 0, 16, alpha, rng)
    Q = strings_from_list([mutate(S.get(int(rng.integers(0, 40_003))), int(rng.integers(0, 4)), alpha, rng)
                           for _ in range(401)])
    ix = gts.Index.build(S, "edit", fanout=20, root_pivot=0)
    s0 = ix.info()["seq"]
    dele = rng.choice(40_003, 900, replace=False)
    ix.delete(dele)
    dl = np.full(40_003, np.iinfo(np.int64).max, np.int64)
    dl[dele] = s0 + np.arange(900)
    ins, qs = np.full(40_003, -1, np.int64), np.full(401, ix.info()["seq"], np.int64)
    r = ix.knn(Q, 6, precision=prec)
    assert r.stats["tiles"] > 0
    off, ids, dist, _ = oracle.knn_query("edit", S, Q, 6, ins, dl, qs)
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.array_equal(r.dist, dist.astype(np.float32))
    radii = np.resize(np.array([0, 1, 2, 5], np.float32), 401)
    r = ix.range(Q, radii, precision=prec)
    off, ids, dist, _ = oracle.range_query("edit", S, Q, radii, ins, dl, qs)
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    assert np.array_equal(r.dist, dist.astype(np.float32))
    ix.close()
