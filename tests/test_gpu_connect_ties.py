"""A full-scan repair among many nodes at one distance: only the nodes that can be the nearest take
part in the final choice, however many others tie behind them, with and without allocation."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


def _noalloc(x, adj, deg, nav):
    b, a, dg, nv = (torch.from_numpy(v).cuda() for v in (x, adj.copy(), deg.copy(), nav))
    rep = ctypes.c_int64(-1)
    rc = ssg.lib().ssg_connect_noalloc(*(ctypes.c_void_p(t.data_ptr()) if not isinstance(t, int) else t
                                         for t in (b, *x.shape, a, dg, a.shape[1], nv, nv.numel())),
                                       ctypes.byref(rep),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, ssg.lib().ssg_last_error()
    return a, dg, rep.value


@pytest.mark.parametrize("call", ["connect", "noalloc"])
@pytest.mark.parametrize("n,near", [(3_000, 1), (60_000, 2), (300_000, 1), (300_000, 3000)])
def test_repairs_behind_many_ties(n, near, call):
    """A tree over all but the last four nodes, which lie at the origin; `near` nodes of the tree lie
    at distance 1 of it and all the others at distance 3."""
    R, m = 6, n - 4
    x = np.zeros((n, 4), np.float32)
    x[:m, 0] = 3
    x[np.random.default_rng(n).choice(np.arange(m // 2, m), near, replace=False), 0] = 1
    i = np.arange(n, dtype=np.int64)[:, None]
    adj = 4 * i + 1 + np.arange(4)[None]
    deg = np.clip(m - (4 * i[:, 0] + 1), 0, 4).astype(np.int32)
    deg[m:] = 0
    adj = np.where(np.arange(R)[None] < deg[:, None], np.pad(adj, ((0, 0), (0, R - 4))), -1).astype(np.int32)
    nav = np.asarray([0], np.int32)
    want = oracle.connect(x, adj, deg, nav)
    a, g, rep = ssg.connect(x, adj, deg, torch.from_numpy(nav)) if call == "connect" else _noalloc(x, adj, deg, nav)
    assert rep == want[2] == 4
    assert np.array_equal(g.cpu().numpy(), want[1])
    assert np.array_equal(a.cpu().numpy(), want[0])
