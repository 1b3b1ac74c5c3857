"""Integer queries over byte rows whose length is and is not a multiple of 16 bytes (pieces of 16 bytes
or words, a kernel each): less than one step of the loads, whole steps, and a remainder behind them.
Everything is an integer below 2^24, so ids and distances equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [3, 16, 20, 100, 112, 128, 129, 148, 160, 254])
def test_rows_of_any_length_equal_the_oracle(d):
    rng = np.random.default_rng(d)
    top = 255 if d <= 128 else 150  # 2 d top^2 stays below 2^24: byte rows are kept
    x = np.clip(np.rint(rng.normal(70, 40, size=(1500, d))), 0, top).astype(np.float32)
    q = np.clip(np.rint(rng.normal(70, 40, size=(40, d))), 0, top).astype(np.float32)
    base = torch.from_numpy(x).cuda()
    g = ssg.build(base, 20, 60, 24, 60.0, n_nav=3)
    adj, deg, nav = (t.cpu().numpy() for t in (g.adj, g.deg, g.nav))
    for k, ls in ((1, 10), (10, 70)):
        want, want_d2 = oracle.search(x, adj, deg, nav, q, k, ls)[:2]
        ids, d2 = g.search(base, torch.from_numpy(q).cuda(), k, ls)
        assert np.array_equal(ids.cpu().numpy(), want)
        assert np.array_equal(d2.cpu().numpy(), want_d2.astype(np.float32))
