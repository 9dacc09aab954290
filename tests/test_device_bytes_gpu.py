"""The memory that an index reports covers what its first queries build and keep."""
import numpy as np
import pytest

from synth import ACGT, random_strings, small_vectors

pytestmark = pytest.mark.gpu


def test_tensor_core_rows_and_raw_norms():
    import paper_2404_00966_gb300 as gts
    X, Q = small_vectors(20_000, 40, 200, seed=1)
    for metric in ("l2", "cos"):
        ix = gts.Index.build(X, metric, fanout=20, root_pivot=0)
        before = ix.info()["device_bytes"]
        assert before >= 20_000 * (40 * 4 * (2 if metric == "cos" else 1) + 16)     # rows (and raw rows), ids, marks
        ix.knn(Q, 3, precision="bf16")
        # 64 columns of two bf16 parts, the norm and the residual of a row; its sum of squares under the angle
        grown = 20_000 * (64 * 2 * 2 + 4 + 4 + (8 if metric == "cos" else 0))
        assert ix.info()["device_bytes"] - before >= grown
        ix.close()


def test_string_counts_and_codes():
    import paper_2404_00966_gb300 as gts
    rng = np.random.default_rng(2)
    n, nq = 90_000, 520
    S, Q = random_strings(n, 40, 60, ACGT, rng), random_strings(nq, 40, 60, ACGT, rng)
    ix = gts.Index.build(S, "edit", fanout=20, root_pivot=0)
    before = ix.info()["device_bytes"]
    ix.range(Q, np.full(nq, 5.0, np.float32), precision="bf16")
    assert ix.info()["device_bytes"] - before >= n * (64 + 256)       # 3-gram counts and the tensor cores' codes
    ix.close()
