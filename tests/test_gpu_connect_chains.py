"""Repairs that kNN rows settle, on their longer routes: a row whose first qualifying entry lies in a
later piece of 32 entries or past the 128 kept in registers, islands whose traversals take the whole
block or the grid, and more nodes than the bitmap in shared memory holds.  A replay on the host names
the route; graphs and counts equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


def _islands(seed, d, core, islands, first, neck, far):
    """A cloud of `core` rows and, in random directions, islands of three parts: `first` rows close
    together, whose graph edges stay among them but whose kNN rows reach the cloud, a thin neck of
    rows leading away, and a cloud of `far` rows at its end."""
    rng = np.random.default_rng(seed)
    xs = [rng.standard_normal((core, d))]
    for _ in range(islands):
        u = rng.standard_normal(d)
        u /= np.linalg.norm(u)
        xs.append(rng.standard_normal((first, d)) * 0.1 + 7.5 * u)
        if neck:
            xs.append(rng.standard_normal((neck, d)) * 0.15 + u * np.linspace(8, 16.5, neck)[:, None])
            xs.append(rng.standard_normal((far, d)) + 18.5 * u)
    return np.concatenate(xs).astype(np.float32)


def _replay(x, K, R, nav, adj, deg):
    """The repairs one after another: (places in the rows, largest levels), scans, the graph."""
    knn, _ = oracle.knn_rows(x, K)
    adj, deg, n = adj.copy(), deg.copy(), len(x)
    places, levels, scans = [], [], 0

    def reach(u):
        largest, front = 0, [u]
        reached[u] = True
        while front:
            new = []
            for w in front:
                for y in adj[w, :deg[w]]:
                    if not reached[y]:
                        reached[y] = True
                        new.append(y)
            front, largest = new, max(largest, len(new))
        return largest

    for s in nav:
        reached = np.zeros(n, bool)
        reach(s)
        while not reached.all():
            u = int(np.argmin(reached))
            at = np.flatnonzero(reached[knn[u]] & (deg[knn[u]] < R))
            if len(at):
                v = knn[u][at[0]]
            else:
                ok = np.flatnonzero(reached & (deg < R))
                d2 = ((x[ok].astype(np.float64) - x[u]) ** 2).sum(1)
                v = ok[np.lexsort((ok, d2))[0]]
                scans += 1
            adj[v, deg[v]] = u
            deg[v] += 1
            level = reach(u)
            if len(at):
                places.append(at[0])
                levels.append(level)
    return places, levels, scans, adj


@pytest.mark.parametrize("data,K,L,R,place,level", [
    ((3, 6, 1500, 1, 140, 0, 0), 180, 30, 8, 129, 0),      # past the pieces in registers
    ((4, 6, 1500, 2, 140, 0, 0), 200, 30, 6, 129, 0),
    ((0, 3, 1500, 1, 80, 40, 3000), 200, 40, 24, 64, 257),   # a level that the block takes
    ((1, 4, 1500, 1, 100, 30, 3000), 200, 60, 32, 96, 513),
    ((2, 6, 1500, 4, 100, 40, 300), 200, 40, 24, 64, 33),
])
def test_rows_and_levels_equal_the_oracle(data, K, L, R, place, level):
    x = _islands(*data)
    nav = np.asarray([5, 7], np.int32)
    ref = oracle.build_graph(x, K, L, R, 60.0, nav)
    places, levels, scans, adj = _replay(x, K, R, nav, ref["adj1"], ref["deg1"])
    assert np.array_equal(adj, ref["adj"])
    assert max(places) >= place and max(levels) >= level      # the routes this case is for
    g = ssg.build(x, K, L, R, 60.0, nav=nav)
    assert g.stats["n_repair"] == ref["n_repair"] == len(places) + scans
    assert g.stats["n_repair_knn_row"] == len(places)
    assert np.array_equal(g.deg.cpu().numpy(), ref["deg"])
    assert np.array_equal(g.adj.cpu().numpy(), ref["adj"])


def test_bitmap_in_global_memory():
    """1.7M nodes: the bitmap of reached nodes does not fit shared memory."""
    x = np.concatenate([_islands(5, 3, 1500, 3, 60, 30, 400),
                        np.random.default_rng(6).uniform(40, 60, (1_700_000, 3))]).astype(np.float32)
    n, K, L, R = len(x), 120, 30, 16
    nav = np.asarray([n // 2, 9], np.int32)
    b = torch.from_numpy(x).cuda()
    g = ssg.build(b, K, L, R, 60.0, nav=nav)
    ids, _ = ssg.knn(b, K)
    pid, _, plen = ssg.pool(b, ids, L)
    a1, d1 = ssg.reverse(b, *ssg.prune(b, pid, plen, R, 60.0), 60.0)
    adj, deg, rep = oracle.connect(x, a1.cpu().numpy(), d1.cpu().numpy(), nav)
    assert g.stats["n_repair"] == rep and 0 < g.stats["n_repair_knn_row"] < rep
    assert np.array_equal(g.deg.cpu().numpy(), deg)
    assert np.array_equal(g.adj.cpu().numpy(), adj)
