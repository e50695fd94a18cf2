"""Workloads of the framework, for measuring it: each case is one call (or one
short chain of calls) of the public API, as a program that uses it makes them.

    cases = listed()                 # fixed cases
    state = prepare(cases[0], 1)     # graph handle, sources, output buffers
    out = run(state)                 # one pass

Graphs are drawn on the GPU from the seed: R-MAT graphs (a/b/c/d =
0.57/0.19/0.19/0.05, ids permuted, loops and duplicates removed) stand for
social networks, grids with dropped edges and diagonal shortcuts for road
networks. Weights are 1..255 and 100..10000, as in the package's own inputs.
"""
from __future__ import annotations

import math

import torch

from paper_2103_14915_gb300 import fg

ROAD_SSSP = {"sched": fg.FG_SCHED_PRIORITY, "sched_window": 50490, "delta": 25245}  # the tuner's kind of choice on
ROAD_BFS = {"sched": fg.FG_SCHED_PRIORITY, "sched_window": 24}                      # road grids: priority windows
ALPHA = 0.15


def listed():
    return [
        # one route query on a small map: launches and latency are all there is
        {"name": "sssp_tiny", "kind": "sssp", "graph": "grid", "rows": 41, "cols": 48, "nq": 1, "tuned": False},
        # landmark distances on a social network, the framework's headline batch
        {"name": "sssp_powerlaw", "kind": "sssp", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False,
         "nq": 256, "tuned": False},
        # a served batch of requests on a directed (follower) graph, ragged in every size
        {"name": "sssp_directed", "kind": "sssp", "graph": "rmat", "n": 300007, "ef": 24, "directed": True, "nq": 97,
         "tuned": False},
        # hop distances from the same kind of sources
        {"name": "bfs_powerlaw", "kind": "bfs", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False, "nq": 256,
         "tuned": False},
        # a handful of hop queries on a middling graph
        {"name": "bfs_few", "kind": "bfs", "graph": "rmat", "n": 70001, "ef": 16, "directed": False, "nq": 13,
         "tuned": False},
        # distance tables on a road network, with the schedule the tuner picks there
        {"name": "sssp_road", "kind": "sssp", "graph": "grid", "rows": 1024, "cols": 1024, "nq": 256, "tuned": True},
        # hop counts on a road network of odd sides
        {"name": "bfs_road", "kind": "bfs", "graph": "grid", "rows": 701, "cols": 1113, "nq": 100, "tuned": True},
        # personalised PageRank of seed users
        {"name": "ppr_powerlaw", "kind": "ppr", "graph": "rmat", "n": 1 << 18, "ef": 16, "directed": False, "nq": 64,
         "eps": 1e-6},
        # community profile: sweep cuts over the PPR rows of 0.01% of the vertices
        {"name": "ncp_sweep", "kind": "ncp", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False, "nq": 105,
         "top": 4096},
        # landmark labels from 1,024 distance rows, then a million distance estimates
        {"name": "landmarks", "kind": "ll", "n": 1 << 18, "K": 1024, "Q": 1 << 20},
        # betweenness centrality from 100 sampled sources
        {"name": "bc_powerlaw", "kind": "bc", "graph": "rmat", "n": 1 << 17, "ef": 16, "directed": False, "nq": 100},
        # random walks for node embeddings: ten walks of 80 steps for each of 100,000 vertices
        {"name": "walks", "kind": "rw", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False, "nq": 1000000,
         "length": 80},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sssp", "sssp", "sssp", "bfs", "bfs", "ppr", "ncp", "ll", "bc", "rw"])
    if kind == "ll":
        return {"kind": "ll", "n": _log(rng, 1000, 1 << 18), "K": _log(rng, 8, 1024), "Q": _log(rng, 1000, 1 << 20)}
    if kind in ("sssp", "bfs") and rng.random() < 0.4:
        return {"kind": kind, "graph": "grid", "rows": _log(rng, 16, 1024), "cols": _log(rng, 16, 1024),
                "nq": _log(rng, 1, 256), "tuned": rng.random() < 0.7}
    top_n = {"ppr": 1 << 18, "bc": 1 << 17}.get(kind, 1 << 20)
    c = {"kind": kind, "graph": "rmat", "n": _log(rng, 1 << 11, top_n), "ef": rng.choice([8, 12, 16]),
         "directed": False}
    if kind in ("sssp", "bfs"):
        c.update(directed=rng.random() < 0.3, nq=_log(rng, 1, 256), tuned=False)
    elif kind == "ppr":
        c.update(nq=_log(rng, 1, 64), eps=rng.choice([1e-5, 1e-6]))
    elif kind == "ncp":
        c.update(nq=_log(rng, 1, 105), top=_log(rng, 16, 4096))
    elif kind == "bc":
        c.update(nq=_log(rng, 1, 100))
    else:
        c.update(nq=_log(rng, 100, 1000000), length=rng.choice([10, 40, 80]))
    return c


# ---- graphs ------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rmat_edges(n, ef, gen):
    """About ef * n edges: R-MAT cells of the enclosing power of two under permuted ids, those below n kept."""
    scale = max(1, (n - 1).bit_length())
    count = int(ef * n * ((1 << scale) / n) ** 2)
    u = torch.zeros(count, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(scale):
        r = torch.rand(count, device="cuda", generator=gen)
        u.mul_(2).add_(r >= 0.76)
        v.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = torch.randperm(1 << scale, device="cuda", generator=gen)
    u, v = perm[u], perm[v]
    keep = (u < n) & (v < n) & (u != v)
    return u[keep], v[keep]


def _grid_edges(rows, cols, gen):
    """Right and down edges, 5% of them dropped, and a diagonal shortcut at 1% of the vertices."""
    i = torch.arange(rows * cols, device="cuda").view(rows, cols)
    us = [i[:, :-1].flatten(), i[:-1].flatten(), i[:-1, :-1].flatten(), i[1:, :-1].flatten()]
    vs = [i[:, 1:].flatten(), i[1:].flatten(), i[1:, 1:].flatten(), i[:-1, 1:].flatten()]
    us, vs = list(us), list(vs)
    for k, p in enumerate((0.95, 0.95, 0.005, 0.005)):
        keep = torch.rand(us[k].numel(), device="cuda", generator=gen) < p
        us[k], vs[k] = us[k][keep], vs[k][keep]
    return torch.cat(us), torch.cat(vs)


def _csr(case, seed):
    """(n, row_ptr int64, col int32, w int32, arc sources int64) on the GPU; adjacency lists sorted."""
    gen = _gen(seed)
    if case["graph"] == "grid":
        n, (u, v), lo, hi, directed = case["rows"] * case["cols"], _grid_edges(case["rows"], case["cols"], gen), 100, \
            10000, False
    else:
        n, (u, v), lo, hi, directed = case["n"], _rmat_edges(case["n"], case["ef"], gen), 1, 255, case["directed"]
    key = torch.unique(u * n + v if directed else torch.cat([u * n + v, v * n + u]))
    u, v = key // n, key % n
    h = torch.minimum(u, v) * 1000003 + torch.maximum(u, v) * 7919 + seed * 104729  # both arcs of an edge alike
    h = (h ^ (h >> 15)) * 2246822519
    w = lo + ((h ^ (h >> 13)) & 0x7FFFFFFF) % (hi - lo + 1)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return n, row_ptr, v.to(torch.int32), w.to(torch.int32), u


def _sources(case, row_ptr, seed):
    """nq sources with out-arcs; PPR seeds spread over the powers of two of the degree. Repeats where too few are there."""
    gen = _gen(seed + 977)
    deg = row_ptr[1:] - row_ptr[:-1]
    cand = torch.nonzero(deg > 0).flatten()
    k = case["nq"]
    if case["kind"] == "rw":
        pick = torch.randint(cand.numel(), (k,), device="cuda", generator=gen)
    elif case["kind"] == "ppr" and k <= cand.numel():
        b = torch.log2(deg[cand].double()).long()
        pick = torch.multinomial(1.0 / torch.bincount(b)[b].double(), k, generator=gen)
    else:
        pick = torch.randperm(cand.numel(), device="cuda", generator=gen)[torch.arange(k, device="cuda") % cand.numel()]
    return cand[pick].to(torch.int32)


def _ppr_like_rows(case, row_ptr, seed):
    """Rows as PPR leaves them: a part of the vertices has mass, log-normal around the degree's share."""
    gen = _gen(seed + 31)
    deg = (row_ptr[1:] - row_ptr[:-1]).float()
    rows = torch.randn((case["nq"], case["n"]), device="cuda", generator=gen).mul_(1.5).exp_()
    rows *= deg / max(1.0, float(deg.sum()))
    share = torch.rand((case["nq"], 1), device="cuda", generator=gen) * 0.9 + 0.05
    rows *= torch.rand((case["nq"], case["n"]), device="cuda", generator=gen) < share
    return rows


class _Graph:
    """A graph handle of the library, given back with the object."""

    def __init__(self, n, row_ptr, col, w):
        torch.cuda.synchronize()
        st, self.h = fg.fg_graph_create_ex(n, col.numel(), row_ptr, col, w, fg.FG_DEVICE_PTRS,
                                           fg.fg_default_graph_opts())
        fg.check(st)

    def __del__(self):
        if getattr(self, "h", None):
            fg.fg_graph_destroy(self.h)
            self.h = None


def _ll_inputs(case, seed):
    gen = _gen(seed)
    dist = torch.randint(0, 20000, (case["K"], case["n"]), dtype=torch.int32, device="cuda", generator=gen)
    dist.masked_fill_(torch.rand(dist.shape, device="cuda", generator=gen) < 0.005, -1)  # not reached
    pairs = torch.randint(0, case["n"], (case["Q"], 2), dtype=torch.int32, device="cuda", generator=gen)
    return dist, pairs


# ---- one case: prepare, run --------------------------------------------------------

def prepare(case, seed):
    kind, dev = case["kind"], "cuda"
    s = {"case": case, "seed": seed}
    if kind == "ll":
        s["dist"], s["pairs"] = _ll_inputs(case, seed)
        s["labels"] = torch.empty((case["n"], case["K"]), dtype=torch.int32, device=dev)
        s["est"] = torch.empty(case["Q"], dtype=torch.int64, device=dev)
        return s
    n, row_ptr, col, w, _ = _csr(case, seed)
    s["g"] = _Graph(n, row_ptr, col, None if kind in ("ppr", "ncp", "rw") else w)
    nq = case["nq"]
    if kind != "ncp":
        s["src"] = _sources(case, row_ptr, seed)
    if kind in ("sssp", "bfs"):
        s["out"] = torch.empty((nq, n), dtype=torch.int32, device=dev)
        s["opts"] = fg.fg_default_opts(**(ROAD_SSSP if kind == "sssp" else ROAD_BFS)) if case["tuned"] else None
    elif kind == "ppr":
        s["p"] = torch.empty((nq, n), dtype=torch.float32, device=dev)
        s["mass"] = torch.empty(nq, dtype=torch.float64, device=dev)
    elif kind == "ncp":
        s["p"] = _ppr_like_rows(case, row_ptr, seed)
        s["order"] = torch.empty((nq, case["top"]), dtype=torch.int32, device=dev)
        s["phi"] = torch.empty((nq, case["top"]), dtype=torch.float64, device=dev)
        s["count"] = torch.empty(nq, dtype=torch.int32, device=dev)
        s["ncp"] = torch.empty(case["top"], dtype=torch.float64, device=dev)
    elif kind == "bc":
        s["dist"] = torch.empty((nq, n), dtype=torch.int32, device=dev)
        fg.check(fg.fg_sssp_batch(s["g"].h, s["src"], nq, s["dist"]))
        fg.check(fg.fg_sync())
        s["bc"] = torch.empty(n, dtype=torch.float64, device=dev)
    else:
        s["paths"] = torch.empty((nq, case["length"] + 1), dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "sssp":
        fg.check(fg.fg_sssp_batch(s["g"].h, s["src"], case["nq"], s["out"], None, s["opts"]))
        fg.check(fg.fg_sync())
        return s["out"]
    if kind == "bfs":
        fg.check(fg.fg_bfs_batch(s["g"].h, s["src"], case["nq"], s["out"], None, s["opts"]))
        fg.check(fg.fg_sync())
        return s["out"]
    if kind == "ppr":
        fg.check(fg.fg_ppr_batch(s["g"].h, s["src"], case["nq"], ALPHA, case["eps"], s["p"], None, s["mass"]))
        fg.check(fg.fg_sync())
        return {"p": s["p"], "mass": s["mass"]}
    if kind == "ncp":
        fg.check(fg.fg_ncp_sweep(s["g"].h, s["p"], case["nq"], case["top"], s["order"], s["phi"], s["count"],
                                 s["ncp"]))
        return {"order": s["order"], "phi": s["phi"], "count": s["count"], "ncp": s["ncp"]}
    if kind == "ll":
        fg.check(fg.fg_ll_build_labels(s["dist"], case["K"], case["n"], s["labels"]))
        fg.check(fg.fg_ll_query(s["labels"], case["n"], case["K"], s["pairs"], case["Q"], s["est"]))
        return {"labels": s["labels"], "est": s["est"]}
    if kind == "bc":
        st, info = fg.fg_bc_accumulate(s["g"].h, s["src"], case["nq"], s["dist"], True, s["bc"])
        fg.check(st)
        return {"bc": s["bc"], "waves": int(info.waves), "sigma_max": float(info.sigma_max)}
    fg.check(fg.fg_rw_batch(s["g"].h, s["src"], case["nq"], case["length"], s["seed"], s["paths"]))
    return s["paths"]


def work(case):
    """Each input read once, each output written once; arcs counted before duplicates are removed."""
    kind = case["kind"]
    if kind == "ll":
        n, K, Q = case["n"], case["K"], case["Q"]
        return {"bytes": 8 * K * n + 4 * K * min(n, 2 * Q) + 16 * Q, "flops": 2 * K * Q}
    n = case["n"] if case["graph"] == "rmat" else case["rows"] * case["cols"]
    arcs = 4 * n if case["graph"] == "grid" else case["ef"] * n * (1 if case["directed"] else 2)
    nq, graph = case["nq"], 4 * n + 4 * arcs
    if kind == "sssp":  # one sum per arc and query
        return {"bytes": graph + 4 * arcs + 4 * nq * n, "flops": nq * arcs}
    if kind == "bfs":
        return {"bytes": graph + 4 * nq * n, "flops": nq * arcs}
    if kind == "ppr":  # every vertex with mass above the threshold pushes at least once
        return {"bytes": graph + 4 * nq * n, "flops": 2 * nq * arcs}
    if kind == "ncp":
        return {"bytes": 4 * nq * n + 4 * n + 12 * nq * case["top"], "flops": 2 * nq * n}
    if kind == "bc":
        return {"bytes": graph + 4 * arcs + 4 * nq * n + 8 * n, "flops": 2 * nq * arcs}
    return {"bytes": nq * (4 * (case["length"] + 1) + 12 * case["length"]), "flops": nq * case["length"]}


# ---- exact values, in plain torch ----------------------------------------------------

def _exact_rows(case, n, row_ptr, col, w, u, src):
    """Distances (w given) or levels by rounds over the arcs sorted by their target; float64 holds them exactly."""
    order = torch.argsort(col.long(), stable=True)
    frm, wt = u[order], (w[order].double() if w is not None else torch.ones(order.numel(), device="cuda").double())
    into = torch.bincount(col.long(), minlength=n)
    out = torch.empty((src.numel(), n), dtype=torch.int32, device="cuda")
    for q in range(0, src.numel(), 16):
        s = src[q:q + 16].long()
        d = torch.full((n, s.numel()), math.inf, dtype=torch.float64, device="cuda")
        d[s, torch.arange(s.numel(), device="cuda")] = 0.0
        while True:
            via = torch.segment_reduce(d[frm] + wt[:, None], "min", lengths=into, axis=0, initial=math.inf, unsafe=True)
            new = torch.minimum(d, via)
            if torch.equal(new, d):
                break
            d = new
        out[q:q + 16] = torch.where(torch.isinf(d), -1.0, d).T.to(torch.int32)
    return out


def _exact_ppr(n, row_ptr, col, src):
    deg = (row_ptr[1:] - row_ptr[:-1]).double()
    adj = torch.sparse_csr_tensor(row_ptr, col.long(), torch.ones(col.numel(), dtype=torch.float64, device="cuda"),
                                  (n, n))
    e = torch.zeros((n, src.numel()), dtype=torch.float64, device="cuda")
    e[src.long(), torch.arange(src.numel(), device="cuda")] = 1.0
    x = e * ALPHA
    for _ in range(200):  # 0.85^200 < 1e-14; both arcs of an edge are there, so adj is its own transpose
        x = ALPHA * e + (1 - ALPHA) * (adj @ (x / deg.clamp(min=1.0)[:, None]))
    return x.T.contiguous()


def _arcs_of(row_ptr, v):
    """(owner position, arc index) of every arc of the vertices v."""
    cnt = row_ptr[v + 1] - row_ptr[v]
    own = torch.repeat_interleave(torch.arange(v.numel(), device=v.device), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    return own, torch.arange(own.numel(), device=v.device) - first[own] + row_ptr[v][own]


def _exact_ncp(case, n, row_ptr, col, p):
    nq, top, m = case["nq"], case["top"], col.numel()
    deg = row_ptr[1:] - row_ptr[:-1]
    order = torch.full((nq, top), -1, dtype=torch.int32, device="cuda")
    phi = torch.full((nq, top), math.nan, dtype=torch.float64, device="cuda")
    count = torch.zeros(nq, dtype=torch.int32, device="cuda")
    for q in range(nq):
        key = torch.where(p[q] > 0, p[q] / deg.clamp(min=1).float(), torch.full_like(p[q], -1.0))
        v = torch.sort(key, descending=True, stable=True).indices[: min(top, int((p[q] > 0).sum()))]
        k = v.numel()
        rank = torch.full((n,), n, dtype=torch.int64, device="cuda")
        rank[v] = torch.arange(k, device="cuda")
        own, e = _arcs_of(row_ptr, v)
        inside = torch.bincount(own[rank[col[e].long()] < own], minlength=k)
        cut, vol = torch.cumsum(deg[v] - 2 * inside, 0), torch.cumsum(deg[v], 0)
        den = torch.minimum(vol, m - vol)
        order[q, :k], count[q] = v.to(torch.int32), k
        phi[q, :k] = torch.where(den > 0, cut.double() / den.clamp(min=1).double(), 1.0)
    ncp = torch.where(torch.isnan(phi), math.inf, phi).amin(0)
    return {"order": order, "phi": phi, "count": count, "ncp": ncp}


def _exact_bc(case, n, row_ptr, col, w, u, src):
    """Brandes' sums: path counts by number of hops, dependencies by rounds until they stand."""
    dist = _exact_rows(case, n, row_ptr, col, w, u, src).long()
    bc = torch.zeros(n, dtype=torch.float64, device="cuda")
    waves, most = 0, 0.0
    for q in range(src.numel()):
        d = dist[q]
        on = (d[u] >= 0) & (d[u] + w.long() == d[col.long()])
        a, b = u[on], col[on].long()
        at = torch.zeros(n, dtype=torch.float64, device="cuda")
        at[src[q].long()] = 1.0
        sigma, hops = at.clone(), 0
        while True:
            at = torch.zeros_like(at).index_add_(0, b, at[a])
            hops += 1
            if not bool(at.any()):
                break
            sigma += at
        share, delta = sigma[a] / sigma[b], torch.zeros_like(sigma)
        for _ in range(hops):
            delta = torch.zeros_like(sigma).index_add_(0, a, share * (1 + delta[b]))
        delta[src[q].long()] = 0.0
        bc += delta
        waves, most = max(waves, hops), max(most, float(sigma[d > 0].max()) if bool((d > 0).any()) else 0.0)
    return {"bc": bc, "waves": waves, "sigma_max": most}


def _exact_walks(case, n, row_ptr, col, src, seed):
    def const(x):
        return x - (1 << 64) if x >= 1 << 63 else x

    def shr(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)

    out = torch.empty((case["nq"], case["length"] + 1), dtype=torch.int32, device="cuda")
    at = src.long()
    out[:, 0] = src
    q = torch.arange(case["nq"], device="cuda") << 32
    for t in range(case["length"]):
        z = seed + (q + (t + 1)) * const(0x9E3779B97F4A7C15)
        z = (z ^ shr(z, 30)) * const(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * const(0x94D049BB133111EB)
        z = z ^ shr(z, 31)
        here = at.clamp(min=0)
        d = row_ptr[here + 1] - row_ptr[here]
        safe = d.clamp(min=1)
        r = (shr(z, 1) % safe * 2 + (z & 1)) % safe  # the 64 bits taken as an unsigned number
        step = col[(row_ptr[here] + r).clamp(max=col.numel() - 1)].long()
        at = torch.where((at < 0) | (d == 0), -1, step)
        out[:, t + 1] = at.to(torch.int32)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "ll":
        dist, pairs = _ll_inputs(case, seed)
        labels = dist.T.contiguous()
        est = torch.empty(case["Q"], dtype=torch.int64, device="cuda")
        for i in range(0, case["Q"], 1 << 16):
            x, y = (labels[pairs[i:i + (1 << 16), k].long()].long() for k in (0, 1))
            both = torch.where((x < 0) | (y < 0), (1 << 62), x + y).amin(1)
            est[i:i + (1 << 16)] = torch.where(both == (1 << 62), -1, both)
        return {"labels": labels, "est": est}
    if kind in ("sssp", "bfs") and case["graph"] == "grid" and case["rows"] * case["cols"] * case["nq"] > 1 << 18:
        return None  # thousands of rounds
    n, row_ptr, col, w, u = _csr(case, seed)
    if kind == "ncp":
        return _exact_ncp(case, n, row_ptr, col, _ppr_like_rows(case, row_ptr, seed))
    src = _sources(case, row_ptr, seed)
    if kind == "sssp":
        return _exact_rows(case, n, row_ptr, col, w, u, src)
    if kind == "bfs":
        return _exact_rows(case, n, row_ptr, col, None, u, src)
    if kind == "ppr":
        return {"p": _exact_ppr(n, row_ptr, col, src),
                "mass": torch.ones(case["nq"], dtype=torch.float64, device="cuda")}
    if kind == "bc":
        return _exact_bc(case, n, row_ptr, col, w, u, src)
    return _exact_walks(case, n, row_ptr, col, src, seed)
