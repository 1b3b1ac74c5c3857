"""The block prune at the edges of its launch classes: rows of up to 128, 256, 512 and 1,024 values, few
and many kept vectors (three or two blocks per SM, kept vectors in shared memory or spilled), pools
shorter than a window and of no multiple of it.  Kept edges equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [96, 128, 129, 200, 256, 257, 300, 384, 420, 512, 513, 1024])
@pytest.mark.parametrize("L,R", [(5, 3), (61, 16), (150, 50), (200, 128)])
def test_prune_equals_the_oracle(d, L, R):
    rng = np.random.default_rng(d + L)
    x = (rng.standard_normal((400, d)) * np.arange(1, d + 1) ** -0.3).astype(np.float32)
    ids, _ = oracle.knn_rows(x, L)
    plen = rng.integers(0, L + 1, size=len(x)).astype(np.int32)
    plen[::7] = L
    ids = np.where(np.arange(L)[None] < plen[:, None], ids, -1).astype(np.int32)
    want, wdeg = oracle.prune(x, ids, plen, R, 75.0)
    adj, deg = ssg.prune(torch.from_numpy(x).cuda(), torch.from_numpy(ids).cuda(), torch.from_numpy(plen).cuda(), R, 75.0)
    assert np.array_equal(deg.cpu().numpy(), wdeg)
    assert np.array_equal(adj.cpu().numpy(), want)
