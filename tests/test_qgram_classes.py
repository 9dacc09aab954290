"""The 3-gram count bound with the functions that the kernels use (qgram.cuh,
compiled for the CPU): L1 distance of the bucket counts <= 6 x edit distance, also
of the counts cut to the levels of the tensor-core filter's code; and, on the
GPU, that the letter classes fit the indexed strings."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from synth import ACGT, LOWER, mutate, random_strings, strings_from_list

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_00966_gb300", "csrc")
SHIM = """
#include "qgram.cuh"
extern "C" void classes(const uint32_t *n, const uint8_t *o, uint8_t *c) { gts::letter_classes(n, o, c); }
extern "C" void counts(const uint8_t *s, int64_t n, const uint8_t *c, uint8_t *h) { gts::qgram_counts(s, n, c, h); }
extern "C" int levels(int b) { return gts::code_levels(b); }
"""
ALPHABETS = {"acgt": ACGT, "lower": LOWER, "01": np.frombuffer(b"01", np.uint8), "ab": np.frombuffer(b"ab", np.uint8),
             "digits": np.frombuffer(b"0123456789", np.uint8), "Aa": np.frombuffer(b"AaCcGgTt", np.uint8),
             "bytes": np.arange(256).astype(np.uint8)}


@pytest.fixture(scope="module")
def grams(tmp_path_factory):
    d = tmp_path_factory.mktemp("qgram")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-x", "c++", str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    L = ctypes.CDLL(str(d / "shim.so"))

    def classes(data):
        n = np.bincount(np.frombuffer(data, np.uint8), minlength=256).astype(np.uint32)
        order = np.lexsort((np.arange(256), -n.astype(np.int64))).astype(np.uint8)
        cls = np.zeros(256, np.uint8)
        L.classes(n.ctypes.data_as(ctypes.c_void_p), order.ctypes.data_as(ctypes.c_void_p),
                  cls.ctypes.data_as(ctypes.c_void_p))
        return cls

    def counts(s, cls):
        h = np.zeros(64, np.uint8)
        L.counts(ctypes.c_char_p(s), ctypes.c_int64(len(s)), cls.ctypes.data_as(ctypes.c_void_p),
                 h.ctypes.data_as(ctypes.c_void_p))
        return h.astype(np.int64)
    cap = np.array([L.levels(b) for b in range(64)], np.int64)
    return classes, counts, cap


@pytest.mark.parametrize("name", sorted(ALPHABETS))
def test_bound_of_the_kernels_counts(grams, name):
    oracle.build()
    classes, counts, cap = grams
    assert cap.sum() == 249 and cap.min() == 3 and cap.max() == 4
    rng = np.random.default_rng(len(name))
    alpha = ALPHABETS[name]
    S = random_strings(200, 0, 120, alpha, rng)
    cls = classes(S.data.tobytes())
    pairs = [(S.get(i), S.get((i * 7 + 1) % S.n)) for i in range(S.n)]
    pairs += [(S.get(i), mutate(S.get(i), int(rng.integers(0, 9)), alpha, rng)) for i in range(S.n)]
    one = bytes(alpha[:1])
    pairs += [(one * 400, one * 380 + bytes(alpha[1:2]) * 3), (b"", bytes(alpha[:2]) + one), (one * 2, one * 3)]
    for a, b in pairs:
        d = oracle.edit_full(a, b)
        ha, hb = counts(a, cls), counts(b, cls)
        assert ha.sum() == min(max(len(a) - 2, 0), ha.sum() if ha.max() == 255 else 10**9)
        assert np.abs(ha - hb).sum() <= 6 * d
        assert np.abs(np.minimum(ha, cap) - np.minimum(hb, cap)).sum() <= 6 * d


def test_classes_split_the_letters(grams):
    classes, _, _ = grams
    assert sorted(classes(b"ACGT" * 9)[ACGT]) == [0, 1, 2, 3]
    assert len(set(classes(b"0100110")[[48, 49]])) == 2
    load = np.bincount(classes(b"0123456789" * 8)[np.arange(48, 58)], minlength=4)
    assert load.max() - load.min() == 1


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["01", "digits", "Aa", "acgt", "lower"])
def test_filter_keeps_no_more_than_hashed_3_grams(name):
    """Pairs that go to the distance: no more than a multiplicative hash of the
    letters into as many buckets lets through (5 % on top: it may spread many
    letters a little better)."""
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(5)
    alpha = ALPHABETS[name]
    base = random_strings(60, 70, 70, alpha, rng)
    S = strings_from_list([mutate(base.get(i % 60), 4, alpha, rng) for i in range(9000)])
    Q = strings_from_list([mutate(base.get(i % 60), 4, alpha, rng) for i in range(120)])
    ix = gts.Index.build(S, "edit", n_pivots=1, fanout=20, root_pivot=0)
    r = ix.range(Q, np.full(120, 7.0, np.float32), precision="bf16")
    off, ids, _, _ = oracle.range_query("edit", S, Q, np.full(120, 7.0, np.float32))
    assert np.array_equal(r.offsets, off) and np.array_equal(r.ids, ids)
    ix.close()

    def hashed(T):
        out = np.zeros((T.n, 64), np.int16)
        for i in range(T.n):
            s = np.frombuffer(T.get(i), np.uint8).astype(np.uint64)
            x = ((s[:-2] << np.uint64(16)) | (s[1:-1] << np.uint64(8)) | s[2:]) * np.uint64(0x9E3779B1) & np.uint64(0xFFFFFFFF)
            out[i] = np.bincount((x >> np.uint64(26)).astype(np.int64), minlength=64)
        return out
    hs, hq = hashed(S), hashed(Q)
    kept = sum(int((np.abs(hs - q).sum(1) <= 42).sum()) for q in hq)
    assert r.stats["candidates"] <= 1.05 * kept, (r.stats["candidates"], kept)
