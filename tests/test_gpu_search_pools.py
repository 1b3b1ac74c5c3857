"""Alg. 1 at the sizes where its pool can go wrong: one entry, around multiples of 32, the largest;
rows of up to 128 neighbours; a batch smaller and larger than the chip; byte and float rows.  Integer
data, so ids and distances equal the oracle's search on the same graph."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    rng = np.random.default_rng(11)
    x = np.clip(np.rint(rng.normal(90, 40, size=(4000, 20))), 0, 255).astype(np.float32)
    base = torch.from_numpy(x).cuda()
    g = ssg.build(base, 60, 300, 128, 85.0, n_nav=11)
    q = np.clip(np.rint(rng.normal(90, 40, size=(300, 20))), 0, 255).astype(np.float32)
    return x, base, g, q


@pytest.mark.parametrize("k,ls", [(1, 1), (1, 2), (5, 31), (32, 32), (10, 33), (64, 64), (10, 65),
                                  (100, 257), (200, 1024)])
@pytest.mark.parametrize("nq", [1, 300])
def test_pool_sizes_equal_the_oracle(case, k, ls, nq):
    x, base, g, q = case
    adj, deg, nav = (t.cpu().numpy() for t in (g.adj, g.deg, g.nav))
    want, _ = oracle.search(x, adj, deg, nav, q[:nq], k, ls)[:2]
    qd = torch.from_numpy(q[:nq]).cuda()
    ids, d2 = g.search(base, qd, k, ls)                                     # byte rows
    assert np.array_equal(ids.cpu().numpy(), want)
    fids, fd2 = ssg.search_adj(base, g.adj, g.deg, g.nav, qd, k, ls)        # float rows
    assert torch.equal(fids, ids) and torch.equal(fd2, d2)
