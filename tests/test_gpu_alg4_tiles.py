"""Alg. 4's pools with a tile limit: a row block's rows are compared with the points of exactly the
pool_tiles 128-point tiles that its list names (rows of more than 128 values: 256-point tiles for
blocks of 128 rows).  Groups of rows far apart make the cluster order, and so every list, known
beforehand; integer data, so the graph equals the oracle's on those pools."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg, synth

pytestmark = pytest.mark.gpu

GROUPS = 16  # the smallest number of clusters: one per group


def _tiles(x, g, block_rows, tile, walk):
    """The points that each block of rows is compared with.  Group c is cluster c and takes the
    stored positions c g .. c g + g - 1; a block goes by the cluster of its middle row."""
    n = len(x)
    centre = x.reshape(GROUPS, g, -1).astype(np.float64).mean(1)
    out = []
    for mid in range(block_rows // 2, n + block_rows // 2, block_rows):
        c = min(mid, n - 1) // g
        d2 = ((centre - centre[c]) ** 2).sum(1)
        d2[c] = -1.0
        seen = []
        for o in np.argsort(d2, kind="stable"):
            for t in range(o * g // tile, (o * g + g - 1) // tile + 1):
                if t not in seen:
                    seen.append(t)
        out.append(np.concatenate([np.arange(t * tile, min(n, t * tile + tile)) for t in seen[:walk]]))
    return out


@pytest.mark.parametrize("n,d,tiles,L", [
    (256, 24, 1, 60),                       # less than one work item, half a tile of its columns
    (1024, 24, 1, 200), (1024, 24, 3, 200),
    (2048, 100, 2, 300), (2048, 128, 5, 90),
    (1024, 130, 1, 300), (1024, 130, 3, 300),   # 128-row blocks, 256-point tiles
    (2048, 200, 2, 100),
])
def test_pools_come_from_the_listed_tiles(n, d, tiles, L):
    rng = np.random.default_rng(n + d + tiles)
    g = n // GROUPS
    centre = rng.integers(10, 190, size=(GROUPS, d))
    x = (np.repeat(centre, g, 0) + rng.integers(-4, 5, size=(n, d))).astype(np.float32)
    block_rows, tile, walk = (256, 128, tiles) if d <= 128 else (128, 256, (tiles + 1) // 2)
    lists = _tiles(x, g, block_rows, tile, walk)
    ids = np.full((n, L), -1, np.int32)
    plen = np.zeros(n, np.int32)
    for i in range(n):
        cand = lists[i // block_rows]
        cand = cand[cand != i]
        d2 = ((x[cand] - x[i]) ** 2).sum(1)
        cand = cand[np.lexsort((cand, d2))][:L]
        ids[i, :len(cand)], plen[i] = cand, len(cand)
    R, alpha, nav = 24, 60.0, synth.nav_ids(n, 3, 5)
    adj0, deg0 = oracle.prune(x, ids, plen, R, alpha)
    adj1, deg1 = oracle.reverse(x, adj0, deg0, alpha)
    adj, deg, _ = oracle.connect(x, adj1, deg1, nav)
    got = ssg.build(torch.from_numpy(x).cuda(), 10, L, R, alpha, nav=nav, pool_tiles=tiles)
    assert np.array_equal(got.deg.cpu().numpy(), deg)
    assert np.array_equal(got.adj.cpu().numpy(), adj)
