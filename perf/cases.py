"""Workloads by which the speed of the library is followed: what users of the index have it do,
through the public binding (paper_1907_06146_gb300/ssg.py), over the sizes they do it at.

A case names a kind of work and its sizes:

* ``search``  a batch of queries against a built index (Alg. 1): one lookup at a time, or a
  batch; byte rows (0..255 integer data) or float rows.
* ``serve``   a burst of mixed host requests (own batch size, k and L_search each) through the
  continuous-batching server.
* ``build``   one whole index (Alg. 3).  Alg. 4's pools are left out: their k-means order, and
  with it the graph, differs from run to run, so their outputs cannot be compared.
* ``many``    independent indices of different shapes built together (multi-tenant).
* ``truth``   brute-force ground truth of a query batch, as taken to measure recall.
* ``stages``  the staged calls in a row: exact kNN graph, pools, prune, reverse merge,
  connectivity, as a program does that inspects or replaces one of them.

Data are drawn on the GPU from the seed, shaped as the project's own generators (synth.py)
shape them: ``sift`` (integers 0..255, about 30% zeros), ``gist`` (non-negative floats in
[0, 1], wide rows), ``deep`` (L2-normalised floats), ``mix`` (16 isotropic Gaussians).
"""
import math

import numpy as np
import torch

from paper_1907_06146_gb300 import ssg

ALPHA = 60.0


def listed():
    return [
        # one lookup against a resident index: an interactive query, all latency
        dict(name="search_one", kind="search", data="sift", n=200_000, d=128, nq=1, k=10, ls=40),
        # the offline batch at recall@10 0.95: the project's headline search workload
        dict(name="search_sift_1m", kind="search", data="sift", n=1_000_000, d=128, nq=10_000,
             k=10, ls=40),
        # float rows, long result lists: the upper end of the serving mix (k = 100, L_search 256)
        dict(name="search_deep", kind="search", data="deep", n=300_000, d=96, nq=4_096, k=100,
             ls=256),
        # a burst of 48 host requests of 1-1,024 queries, k in {1, 10, 100}, L_search in [k, 512]
        dict(name="serve_mixed", kind="serve", data="deep", n=200_000, d=96, requests=48,
             most=1_024),
        # the small configuration: 10,000 float rows of 32 values, where launches count
        dict(name="build_small", kind="build", data="mix", n=10_000, d=32, K=20, L=100, R=32,
             nav=3),
        # the headline build: 1M SIFT-shaped rows with the paper's SIFT1M parameters
        dict(name="build_sift_1m", kind="build", data="sift", n=1_000_000, d=128, K=200, L=100,
             R=50, nav=10),
        # wide float rows with the paper's GIST1M parameters
        dict(name="build_gist_100k", kind="build", data="gist", n=100_000, d=960, K=100, L=500,
             R=70, nav=10),
        # float rows of SIFT's width, larger pools (one index of the multi-tenant batch)
        dict(name="build_mix_200k", kind="build", data="mix", n=200_000, d=128, K=100, L=200,
             R=32, nav=10),
        # an ordinary index of integer rows: a shard, or a collection of its own
        dict(name="build_sift_60k", kind="build", data="sift", n=60_000, d=128, K=200, L=100,
             R=50, nav=10),
        # multi-tenant: six indices of 10,000-80,000 rows, d in {64, 96, 128, 256}, L 100 or 200
        dict(name="build_many", kind="many", count=6, least=10_000, most=80_000, shapes=7),
        # ground truth of 10,000 queries over 1M rows
        dict(name="truth_1m", kind="truth", data="sift", n=1_000_000, d=128, nq=10_000, k=100),
        # the staged calls on rows and counts that no tile divides
        dict(name="stages_ragged", kind="stages", data="mix", n=30_011, d=100, K=50, L=120, R=40,
             nav=5, prec="auto"),
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], even over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("search", "search", "serve", "build", "build", "build", "many", "truth",
                       "stages", "stages"))
    if kind == "search":
        data = rng.choice(("sift", "deep", "mix"))
        k = rng.choice((1, 10, 100))
        return dict(kind=kind, data=data, n=_spread(rng, 10_000, 1_000_000 if data == "sift" else 200_000),
                    d={"sift": 128, "deep": 96, "mix": rng.choice((32, 61, 100, 128, 200))}[data],
                    nq=_spread(rng, 1, 10_000), k=k, ls=_spread(rng, max(k, 10), 512))
    if kind == "serve":
        return dict(kind=kind, data="deep", n=_spread(rng, 10_000, 300_000), d=96,
                    requests=rng.randrange(4, 64), most=_spread(rng, 16, 2_048))
    if kind == "build":
        data = rng.choice(("sift", "gist", "mix", "deep"))
        if data == "sift":
            return dict(kind=kind, data=data, n=_spread(rng, 10_000, 900_000), d=128, K=200, L=100,
                        R=50, nav=10)
        if data == "gist":
            return dict(kind=kind, data=data, n=_spread(rng, 5_000, 90_000), d=960, K=100, L=500,
                        R=70, nav=10)
        if data == "mix":
            return dict(kind=kind, data=data, n=_spread(rng, 5_000, 180_000),
                        d=rng.choice((32, 50, 64, 96, 111, 128, 256)), K=rng.choice((20, 64, 100)),
                        L=rng.choice((100, 150, 200)), R=rng.choice((24, 32, 50)), nav=10)
        return dict(kind=kind, data=data, n=_spread(rng, 10_000, 200_000), d=96, K=100, L=100,
                    R=32, nav=10)
    if kind == "many":
        return dict(kind=kind, count=rng.randrange(2, 8), least=8_000,
                    most=_spread(rng, 20_000, 90_000), shapes=rng.randrange(1_000))
    if kind == "truth":
        data = rng.choice(("sift", "mix"))
        return dict(kind=kind, data=data, n=_spread(rng, 10_000, 1_000_000 if data == "sift" else 200_000),
                    d=128 if data == "sift" else rng.choice((32, 77, 96, 128)),
                    nq=_spread(rng, 1, 9_000), k=rng.choice((1, 10, 100)))
    return dict(kind="stages", data=rng.choice(("mix", "sift")), n=_spread(rng, 2_000, 60_000),
                d=rng.randrange(17, 200), K=rng.randrange(16, 128), L=rng.randrange(40, 200),
                R=rng.randrange(20, 70), nav=rng.randrange(1, 12),
                prec=rng.choice(("auto", "auto", "fp32")))


# ---- data ------------------------------------------------------------------------------------
def _orthonormal(d, gen):
    a = torch.randn(d, d, generator=gen, device="cuda", dtype=torch.float64).cpu()
    q, r = torch.linalg.qr(a)
    return (q * torch.sign(torch.diagonal(r))).to("cuda", torch.float32)


def _cloud(m, d, clusters, gamma, top, gen, centre_scale=1.0):
    """Anisotropic Gaussians sharing one basis and a power-law spectrum: one continuous cloud."""
    basis = _orthonormal(d, gen)
    spec = top * torch.arange(1, d + 1, device="cuda", dtype=torch.float32) ** -gamma

    def normal(rows):
        return torch.randn(rows, d, generator=gen, device="cuda")

    centres = normal(clusters) * (centre_scale * spec)
    spreads = spec * torch.exp(0.3 * normal(clusters))
    lab = torch.randint(clusters, (m,), generator=gen, device="cuda")
    y = torch.empty(m, d, device="cuda")
    for s in range(0, m, 131_072):
        at = lab[s:s + 131_072]
        y[s:s + 131_072] = (centres[at] + normal(at.numel()) * spreads[at]) @ basis.T
    return y


def _rows(data, m, d, gen):
    if data == "mix":
        centres = 2.0 * torch.randn(16, d, generator=gen, device="cuda")
        lab = torch.randint(16, (m,), generator=gen, device="cuda")
        return centres[lab] + torch.randn(m, d, generator=gen, device="cuda")
    if data == "sift":
        y = _cloud(m, d, 1_000, 1.0, 70.0, gen)
        some = y.reshape(-1)[:4_000_000]
        shift = 0.5 - some.sort().values[int(0.3 * some.numel())]
        return (y + shift).round_().clamp_(0.0, 255.0)
    if data == "gist":
        k = np.arange(1, d + 1, dtype=np.float64)
        top = float(np.sqrt(d / np.sum(k ** (-2.0 * 0.67))))
        y = torch.nn.functional.softplus(_cloud(m, d, 500, 0.67, top, gen, 0.5))
        return y / y.max()
    y = _cloud(m, d, 2_000, 1.4, 1.0, gen)
    return y / y.norm(dim=1, keepdim=True)


def _vectors(case, seed):
    """The base rows and, where the case has any, the queries (drawn from the same cloud)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    nq = case.get("nq", 0)
    x = _rows(case["data"], case["n"] + nq, case["d"], gen)
    return x[:case["n"]].contiguous(), x[case["n"]:].contiguous()


def _requests(case):
    """The burst of a serve case: (queries, k, L_search) of each request."""
    r = np.random.Generator(np.random.PCG64(case["requests"] * 1_009 + case["most"]))
    out = []
    for _ in range(case["requests"]):
        k = int(r.choice([1, 10, 100]))
        out.append((int(round(math.exp(r.uniform(0.0, math.log(case["most"]))))), k,
                    int(round(math.exp(r.uniform(math.log(max(k, 10)), math.log(512)))))))
    return out


def _shapes(case):
    """The indices of a many case: (n, d, L)."""
    r = np.random.Generator(np.random.PCG64(case["shapes"]))
    return [(int(round(math.exp(r.uniform(math.log(case["least"]), math.log(case["most"]))))),
             int(r.choice([64, 96, 128, 256])), int(r.choice([100, 200])))
            for _ in range(case["count"])]


def _index(case, base):
    """The index that a search program keeps."""
    return ssg.build(base, K=100, L=100, R=50 if case["data"] == "sift" else 32, alpha=ALPHA)


# ---- the cases -------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "many":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        state["bases"] = [_rows("mix", n, d, gen) for n, d, _ in _shapes(case)]
        return state
    if kind == "serve":
        todo = _requests(case)
        base, q = _vectors(dict(case, nq=sum(m for m, _, _ in todo)), seed)
        q, at, requests = q.cpu().numpy(), 0, []
        for m, k, ls in todo:
            requests.append((np.ascontiguousarray(q[at:at + m]), k, ls))
            at += m
        state["requests"] = requests
        state["graph"] = _index(case, base)
        state["server"] = ssg.Server(state["graph"], base)
        return state
    state["base"], state["queries"] = _vectors(case, seed)
    if kind == "search":
        state["graph"] = _index(case, state["base"])
    if kind == "stages":
        state["nav"] = torch.from_numpy(ssg.nav_ids(case["n"], case["nav"], int(seed))).cuda()
    return state


def _graph(g):
    return {"adj": g.adj, "deg": g.deg, "nav": g.nav}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "search":
        ids, d2 = state["graph"].search(state["base"], state["queries"], case["k"], case["ls"])
        return {"ids": ids, "d2": d2}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(q, k, ls) for q, k, ls in state["requests"]]
        done = [server.wait(t) for t in tickets]
        return {"ids": np.concatenate([r[0].reshape(-1) for r in done]),
                "d2": np.concatenate([r[1].reshape(-1) for r in done])}
    if kind == "build":
        return _graph(ssg.build(state["base"], case["K"], case["L"], case["R"], ALPHA,
                                n_nav=case["nav"]))
    if kind == "many":
        return [_graph(g) for g in ssg.build_batched(state["bases"], 100,
                                                     [L for _, _, L in _shapes(case)], 32, ALPHA)]
    if kind == "truth":
        ids, d2 = ssg.knn_query(state["base"], state["queries"], case["k"])
        return {"ids": ids, "d2": d2}
    base = state["base"]
    ids, d2 = ssg.knn(base, case["K"], case["prec"])
    pool, pool_d2, pool_len = ssg.pool(base, ids, case["L"])
    adj0, deg0 = ssg.prune(base, pool, pool_len, case["R"], ALPHA)
    adj1, deg1 = ssg.reverse(base, adj0, deg0, ALPHA)
    adj, deg, repairs = ssg.connect(base, adj1, deg1, state["nav"])
    return {"knn": ids, "knn_d2": d2, "pool": pool, "pool_d2": pool_d2, "pool_len": pool_len,
            "adj0": adj0, "deg0": deg0, "adj1": adj1, "deg1": deg1, "adj": adj, "deg": deg,
            "repairs": repairs}


def _search_work(nq, k, ls, d, row_value_bytes, R):
    """Alg. 1 expands at least L_search entries; about two thirds of their edges (degree about
    half of R) lead to a row not seen before."""
    edges = ls * R * 0.5
    return (nq * (edges * (4 + 0.66 * d * row_value_bytes) + 4 * d + 8 * k),
            nq * edges * 0.66 * 2 * d)


def work(case):
    kind = case["kind"]
    if kind == "search":
        b, f = _search_work(case["nq"], case["k"], case["ls"], case["d"],
                            1 if case["data"] == "sift" else 4, 50 if case["data"] == "sift" else 32)
    elif kind == "serve":
        parts = [_search_work(m, k, ls, case["d"], 4, 32) for m, k, ls in _requests(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "build":
        n, d = case["n"], case["d"]
        b = 4 * n * (d + case["R"] + 1)
        f = 2.0 * n * n * d + 2.0 * n * case["L"] * d
    elif kind == "many":
        b = sum(4 * n * (d + 33) for n, d, _ in _shapes(case))
        f = sum(2.0 * n * n * d + 2.0 * n * L * d for n, d, L in _shapes(case))
    elif kind == "truth":
        b = 4 * (case["n"] + case["nq"]) * case["d"] + 8 * case["nq"] * case["k"]
        f = 2.0 * case["nq"] * case["n"] * case["d"]
    else:
        n, d = case["n"], case["d"]
        b = 4 * n * (d + 2 * case["K"] + 2 * case["L"] + 3 * case["R"] + 4)
        f = 2.0 * n * n * d + 2.0 * n * case["L"] * d
    return {"bytes": b, "flops": f}


def _nearest(x, q, k, own):
    """Squared distances of each row of q to its k nearest rows of x in 64 bits, ascending;
    own: q is x, and a row is not its own neighbour."""
    x, q = x.double(), q.double()
    x2, q2 = (x * x).sum(1), (q * q).sum(1)
    out = torch.empty(q.shape[0], k, dtype=torch.float64, device=x.device)
    step = max(1, (1 << 28) // x.shape[0])
    for s in range(0, q.shape[0], step):
        e = min(q.shape[0], s + step)
        d2 = q2[s:e, None] + x2[None, :] - 2.0 * (q[s:e] @ x.T)
        if own:
            d2[torch.arange(e - s, device=x.device), torch.arange(s, e, device=x.device)] = math.inf
        out[s:e] = d2.topk(k, largest=False, sorted=True).values
    return out


def exact(case, seed):
    """The kNN and ground-truth distances; graphs are whole numbers, and the distances that a
    search or a pool returns depend on a graph of the library's own."""
    if case["kind"] == "truth":
        base, q = _vectors(case, seed)
        return {"ids": None, "d2": _nearest(base, q, case["k"], False)}
    if case["kind"] == "stages":
        base, _ = _vectors(case, seed)
        return {"knn_d2": _nearest(base, base, case["K"], True)}
    return None
