"""Connectivity on graphs that take each of its routes: many repairs by the full scan, long chains
of repairs by kNN rows, islands whose traversals outgrow one warp, roots that do not reach the
first one, rows of more than 128 neighbours, and exact ties for a repair's nearest node.  Every
graph and repair count equals the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_06146_gb300 import ssg

pytestmark = pytest.mark.gpu


def _graph(n, R, deg, seed, parts):
    """Random out-edges inside each of `parts` ranges of ids (nothing crosses)."""
    rng = np.random.default_rng(seed)
    adj = np.full((n, R), -1, np.int32)
    dg = np.minimum(rng.integers(0, deg + 1, size=n), R).astype(np.int32)
    edges = np.linspace(0, n, parts + 1).astype(int)
    for s, e in zip(edges[:-1], edges[1:]):
        for i in range(s, e):
            k = min(int(dg[i]), e - s - 1)
            dg[i] = k
            c = rng.choice(e - s - 1, size=k, replace=False) if k else np.empty(0, int)
            c = c + s
            adj[i, :k] = np.where(c >= i, c + 1, c)
    return adj, dg


@pytest.mark.parametrize("n,d,R,deg,parts,integer", [
    (257, 8, 4, 2, 1, False),       # many unreached nodes, full scans
    (1000, 5, 6, 3, 3, False),      # islands, padded rows
    (3000, 16, 8, 6, 2, False),     # an island that one warp does not expand
    (400, 3, 140, 2, 4, True),      # wide rows, exact ties
    (33, 4, 3, 1, 33, True),        # no edges at all: every node a repair
])
def test_connect_equals_the_oracle(n, d, R, deg, parts, integer):
    rng = np.random.default_rng(n + d)
    x = rng.integers(0, 4, size=(n, d)) if integer else rng.standard_normal((n, d))
    x = np.ascontiguousarray(x, np.float32)
    adj, dg = _graph(n, R, deg, n, parts)
    nav = np.asarray([n // 2, 0, n - 1], np.int32)
    want = oracle.connect(x, adj, dg, nav)
    a, g, rep = ssg.connect(x, adj, dg, torch.from_numpy(nav))
    assert np.array_equal(g.cpu().numpy(), want[1])
    got = a.cpu().numpy()
    for i in range(n):
        assert np.array_equal(got[i, :want[1][i]], want[0][i, :want[1][i]])
    assert rep == want[2]


@pytest.mark.parametrize("n,d,centres", [(2000, 12, 40), (4000, 24, 200)])
def test_build_with_islands_equals_the_oracle(n, d, centres):
    """Islands far apart: repairs by kNN rows and, across islands, by the full scan."""
    rng = np.random.default_rng(centres)
    c = rng.standard_normal((centres, d)) * 50
    x = (c[rng.integers(0, centres, n)] + rng.standard_normal((n, d))).astype(np.float32)
    nav = np.asarray([3, n // 2, n - 5], np.int32)
    want = oracle.build_graph(x, 10, 30, 12, 60.0, nav)
    g = ssg.build(x, 10, 30, 12, 60.0, nav=nav)
    assert g.stats["n_repair"] == want["n_repair"]
    deg = g.deg.cpu().numpy()
    assert np.array_equal(deg, want["deg"])
    adj = g.adj.cpu().numpy()
    for i in range(n):
        assert np.array_equal(adj[i, :deg[i]], want["adj"][i, :deg[i]])
