"""The tensor-core kNN at the edges of its tiles (256 columns, 512 rows, 64-value chunks, K-steps of
16), of its row buffers and of the split of columns over the chip; with so many ties that a row's
buffer and the final selection are settled by id; and through its launch options.  Integer data, so
every row is exact: ids and distances equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


def _ints(n, d, hi, seed):
    return np.random.default_rng(seed).integers(0, hi, size=(n, d)).astype(np.float32)


@pytest.mark.parametrize("n,d,K,hi", [
    (2, 1, 1, 9), (3, 40, 2, 9), (255, 16, 20, 200), (256, 17, 32, 200), (257, 64, 31, 200), (511, 65, 33, 200),
    (513, 128, 64, 200), (512, 129, 100, 200), (1025, 8, 700, 200), (770, 300, 12, 100),
    (3000, 4, 40, 2),      # 16 distinct rows: hundreds of ties at every threshold
    (5000, 2, 300, 3),     # more ties than a row buffer holds
    (4097, 33, 201, 50),
])
def test_self_join_equals_the_oracle(n, d, K, hi):
    x = _ints(n, d, hi, n * 7 + d)
    ids, d2 = ssg.knn(x, K, "bf16")
    oid, od2 = oracle.knn_rows(x, K)
    assert np.array_equal(ids.cpu().numpy(), oid)
    assert np.array_equal(d2.cpu().numpy(), od2.astype(np.float32))


@pytest.mark.parametrize("n,nq,d,k,hi", [
    (3000, 1, 128, 1, 200), (20000, 3, 128, 100, 200), (9000, 513, 20, 10, 200),
    (30000, 40, 3, 64, 4),  # shared-out columns, ties across the shares
])
def test_queries_equal_the_oracle(n, nq, d, k, hi):
    x, q = _ints(n, d, hi, n), _ints(nq, d, hi, n + 1)
    ids, d2 = ssg.knn_query(x, q, k, "bf16")
    oid, od2 = oracle.knn_queries(x, q, k)
    assert np.array_equal(ids.cpu().numpy(), oid)
    assert np.array_equal(d2.cpu().numpy(), od2.astype(np.float32))


@pytest.mark.parametrize("option", ["knn_prepass_tiles = 8", "knn_stream_rows = 1"])
def test_launch_options_keep_the_graph(option, tmp_path):
    """A self-join large enough for the near-first order, with and without the option."""
    x = torch.from_numpy(_ints(70_000, 12, 100, 5)).cuda()
    table = tmp_path / "table"
    table.write_text(option + "\n")
    a = ssg.build(x, 24, 40, 16, 60.0, n_nav=2)
    b = ssg.build(x, 24, 40, 16, 60.0, n_nav=2, tune_table=str(table))
    assert torch.equal(a.deg, b.deg) and torch.equal(a.adj, b.adj)
