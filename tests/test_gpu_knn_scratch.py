"""The kNN's row buffers where the device has no room for them: a launch takes fewer rounds of rows,
then fewer shares of the columns, with the same result; at one round of unshared rows the call
reports ENOMEM.  Every scratch allocation of a call is made to fail in turn."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,d,K,tolerated", [
    (50_000, 0, 8, 10, 1),    # 98 blocks of rows: two rounds
    (9_000, 300, 20, 30, 1),  # few queries: the columns are shared out
    (200, 0, 12, 5, 0),       # one tile: nothing to give up
])
def test_failed_row_buffers(n, nq, d, K, tolerated):
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.integers(0, 100, size=(n, d)).astype(np.float32)).cuda()
    q = torch.from_numpy(rng.integers(0, 100, size=(nq, d)).astype(np.float32)).cuda()
    call = (lambda: ssg.knn_query(x, q, K, "bf16")) if nq else (lambda: ssg.knn(x, K, "bf16"))
    ids, d2 = call()
    rows = np.sort(rng.choice(nq or n, 100, replace=False))
    want = oracle.knn_queries(x.cpu().numpy(), q.cpu().numpy()[rows], K) if nq else oracle.knn_rows(x.cpu().numpy(), K, rows=rows)
    assert np.array_equal(ids.cpu().numpy()[rows], want[0])
    passed = []
    for nth in range(1, 41):
        ssg.debug_fail_alloc(nth)
        try:
            i2, e2 = call()
            assert torch.equal(i2, ids) and torch.equal(e2, d2)
            passed.append(nth)
        except ssg.SSGError as e:
            assert e.status == 2 and "injected" in str(e)
        finally:
            ssg.debug_fail_alloc(0)
    last = max(set(range(1, 41)) - set(passed))   # the call's last allocation
    assert last < 40 and sum(p < last for p in passed) == tolerated
