"""The certificate of the bf16 kNN path and its exhaustive fallback at the sizes where they can
go wrong: many exact ties around the K-th distance (more survivors than the K the selection
aims at), rows of one and of several 128-value pieces, K + 8 candidates or fewer, and rows that
no band certifies.  The kNN rows equal the oracle's, ids and float64 distances rounded once."""
import numpy as np
import pytest

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


def _rows(n, d, seed, copies, shift):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((n, d)).astype(np.float32) + np.float32(shift)
    if copies:  # groups of identical rows: exact ties at distance 0 and beyond
        x = x[rng.integers(0, max(1, n // copies), size=n)]
    return np.ascontiguousarray(x)


@pytest.mark.parametrize("n,d,K,copies,shift", [
    (300, 3, 7, 0, 0.0),          # padded rows
    (700, 128, 64, 0, 0.0),       # one register piece exactly
    (700, 129, 33, 0, 0.0),       # one value beyond it
    (900, 61, 40, 90, 0.0),       # 90 copies of each row: ties across the K-th distance
    (1200, 200, 100, 300, 0.0),   # more ties than the survivors' buffer holds
    (800, 96, 50, 0, 400.0),      # far from the origin
    (513, 40, 500, 0, 0.0),       # nearly every row is a neighbour
])
def test_knn_rows_equal_the_oracle(n, d, K, copies, shift):
    x = _rows(n, d, n + d, copies, shift)
    ids, d2 = ssg.knn(x, K, "bf16")
    oid, od2 = oracle.knn_rows(x, K)
    assert np.array_equal(ids.cpu().numpy(), oid)
    assert np.array_equal(d2.cpu().numpy(), od2.astype(np.float32))
