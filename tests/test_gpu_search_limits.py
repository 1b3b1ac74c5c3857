"""The largest rows and pools a search takes, and one step beyond: EINVAL, as it always was, though
the kernel could take fewer queries per block.  Inside, results equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["float", "bytes", "work", "host", "server"])
@pytest.mark.parametrize("d,ls,fits", [(5328, 10, True), (5344, 10, False), (1680, 1024, True),
                                       (1696, 1024, False), (8192, 1, False)])
def test_sizes_at_the_limit(entry, d, ls, fits):
    rng = np.random.default_rng(d)
    n, R, k = 300, 32, 1
    top = 20  # (d top^2 stays exact in fp32)
    x = rng.integers(0, top, size=(n, d)).astype(np.float32)
    q = rng.integers(0, top, size=(5, d)).astype(np.float32)
    b, qd = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
    if entry in ("host", "server"):
        g = ssg.build_host(x, 20, 40, R, 60.0, n_nav=2)[0]
    else:
        g = ssg.build(b, 20, 40, R, 60.0, n_nav=2)
    adj, deg, nav = (t.cpu().numpy() for t in (g.adj, g.deg, g.nav))

    def call():
        if entry == "float":
            return ssg.search_adj(b, g.adj, g.deg, g.nav, qd, k, ls)[0].cpu().numpy()
        if entry == "bytes":
            return g.search(b, qd, k, ls)[0].cpu().numpy()
        if entry == "work":
            return ssg.search_work(b, g.adj, g.deg, g.nav, qd, k, ls)[0].cpu().numpy()
        if entry == "host":
            return g.search_host(q, k, ls)[0]
        s = ssg.Server(g)
        try:
            return s.wait(s.submit(q, k, ls))[0]
        finally:
            s.close()

    if fits or entry == "work":   # a counting call holds two queries at once, not eight
        assert np.array_equal(call(), oracle.search(x, adj, deg, nav, q, k, ls)[0])
    else:
        with pytest.raises(ssg.SSGError) as e:
            call()
        assert e.value.status == 1
