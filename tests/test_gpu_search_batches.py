"""Float rows in batches of every size class that the launch distinguishes: up to 16 queries per SM,
up to 24, up to 32 (all at once where shared memory lets them), more (a warp takes several queries one
after another), and rows or pools so long that an SM holds few warps.  Integer values, so ids and
distances equal the oracle's; every query of a batch is checked."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[61, 128, 200, 960])
def case(request):
    d = request.param
    rng = np.random.default_rng(d)
    centres = rng.integers(20, 90, size=(12, d))
    x = (centres[rng.integers(0, 12, 2500)] + rng.integers(-15, 16, size=(2500, d))).astype(np.float32)
    base = torch.from_numpy(x).cuda()
    g = ssg.build(base, 20, 60, 40, 60.0, n_nav=7)
    q = (centres[rng.integers(0, 12, 12000)] + rng.integers(-20, 21, size=(12000, d))).astype(np.float32)
    return x, base, g, q


@pytest.mark.parametrize("k,ls", [(5, 10), (10, 100), (3, 333)])
@pytest.mark.parametrize("per_sm", [0, 2, 16, 20, 28, 70])
def test_batches_equal_the_oracle(case, per_sm, k, ls):
    x, base, g, q = case
    nq = max(1, per_sm * torch.cuda.get_device_properties(0).multi_processor_count - 3)
    nq = min(nq, len(q), 12_000 if ls <= 100 else 4_300)
    adj, deg, nav = (t.cpu().numpy() for t in (g.adj, g.deg, g.nav))
    want_ids, want_d2 = oracle.search(x, adj, deg, nav, q[:nq], k, ls)[:2]
    ids, d2 = ssg.search_adj(base, g.adj, g.deg, g.nav, torch.from_numpy(q[:nq]).cuda(), k, ls)
    assert np.array_equal(ids.cpu().numpy(), want_ids)
    assert np.array_equal(d2.cpu().numpy(), want_d2.astype(np.float32))
