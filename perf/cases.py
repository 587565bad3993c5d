"""Measured cases: what a user of the library has it do, through its public entry points.

Four kinds of case:

- ``build``: canonical labels of one graph (``build_labels``), copied out whole
  (offsets, hubs, distances, and the tree parents where they were asked for).
  Scale-free graphs (R-MAT, Barabasi-Albert) under the degree ranking and
  road-like grids under sampled betweenness are the two families the method is
  for. Default options throughout, as a caller who passes none; the options
  that change what is computed (parents, a weight range that needs 8-byte tree
  keys) and where the arrays live (device, or host in and host out) vary.
- ``query``: one batch of distance queries against resident labels, in the
  three modes of the query interface (merge, grouped, hub-partitioned), from
  one pair (a lookup) to a million (offline scoring), host or device pairs.
- ``paths``: shortest paths, vertices and all, from labels built with parents.
- ``serve``: a burst of requests of uneven size to a server that holds two label
  sets, every one waited for.

All values are integers, so every result is exact.
"""
import numpy as np
import torch

import paper_1907_00140_gb300 as chl

DEV = "cuda"
INF = 1 << 40

# labels per vertex of the families as measured at one size each: (labels,
# vertices, growth exponent). They set the bytes that a build has to write and,
# for the two ends of a pair, the entries that a query has to look at.
LABELS = {"rmat": (102.0, 174_000, 0.36), "ba": (73.7, 50_000, 0.43), "grid": (136.0, 16_382, 0.43)}


def listed():
    return [
        # the smallest build: a graph of 2,000 vertices, where launches and host round trips count
        {"name": "build-ba2k", "kind": "build", "family": "ba", "n": 2000, "m": 3, "wmax": 100},
        # a build request as it arrives at a service: arrays in host memory, labels back to host memory
        {"name": "build-ba50k-host", "kind": "build", "family": "ba", "n": 50_000, "m": 5, "wmax": 100,
         "host": True},
        # the ordinary scale-free build (social and web graphs)
        {"name": "build-rmat18", "kind": "build", "family": "rmat", "scale": 18, "ef": 16, "wmax": 255},
        # heavy weights (travel times in milliseconds, costs): tree keys of 8 bytes
        {"name": "build-rmat16-wide", "kind": "build", "family": "rmat", "scale": 16, "ef": 16,
         "wmax": 100_000},
        # road network: high diameter, long label lists
        {"name": "build-grid512", "kind": "build", "family": "grid", "side": 512, "samples": 64},
        # road network of a town with route recovery: the parents stored with the labels
        {"name": "build-grid128-parents", "kind": "build", "family": "grid", "side": 128, "samples": 32,
         "parents": True},
        # the largest build
        {"name": "build-rmat21", "kind": "build", "family": "rmat", "scale": 21, "ef": 16, "wmax": 1000},
        # one lookup from host memory: latency
        {"name": "query-1", "kind": "query", "family": "rmat", "scale": 18, "ef": 16, "wmax": 255,
         "pairs": 1, "mode": "merge", "host": True, "skew": 0.0},
        # offline scoring: a million uniform pairs resident on the device
        {"name": "query-1m", "kind": "query", "family": "rmat", "scale": 18, "ef": 16, "wmax": 255,
         "pairs": 1_000_000, "mode": "merge", "host": False, "skew": 0.0},
        # labels held as hub partitions, half of the pairs between well-connected vertices
        {"name": "query-parts", "kind": "query", "family": "ba", "n": 100_000, "m": 7, "wmax": 100,
         "pairs": 200_000, "mode": "parts", "host": False, "skew": 0.5},
        # routes on a road network
        {"name": "paths-grid128", "kind": "paths", "family": "grid", "side": 128, "samples": 32,
         "pairs": 20_000, "max_len": 320},
        # continuous batching: a burst of uneven requests over two label sets
        {"name": "serve-burst", "kind": "serve", "family": "rmat", "scale": 16, "ef": 16, "wmax": 255,
         "n2": 25_000, "requests": 200, "mean_pairs": 40.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "query", "query", "paths", "serve"])
    family = "grid" if kind == "paths" and rng.random() < 0.7 else rng.choice(["rmat", "ba", "grid"])
    if kind == "serve":
        family = "rmat"
    c = {"kind": kind, "family": family}
    if family == "rmat":
        c.update(scale=rng.randint(10, 18), ef=rng.randint(4, 16), wmax=_log_int(rng, 10, 1000))
    elif family == "ba":
        c.update(n=_log_int(rng, 300, 200_000), m=rng.randint(3, 8), wmax=_log_int(rng, 10, 1000))
    else:
        c.update(side=_log_int(rng, 12, 330), samples=rng.choice([16, 32]))
    if kind == "build":
        if rng.random() < 0.3 and family != "grid":
            c["wmax"] = _log_int(rng, 50_000, 1_000_000)
        if rng.random() < 0.25:
            c["parents"] = True
        if rng.random() < 0.3:
            c["host"] = True
    elif kind == "query":
        c.update(pairs=_log_int(rng, 1, 1_000_000), mode=rng.choice(["merge", "merge", "grouped", "parts"]),
                 host=rng.random() < 0.4, skew=rng.choice([0.0, 0.5]))
    elif kind == "paths":
        c.update(pairs=_log_int(rng, 1, 50_000), max_len=rng.choice([64, 320, 700]))
    else:
        c.update(scale=rng.randint(10, 16), n2=_log_int(rng, 2000, 50_000), requests=_log_int(rng, 10, 400),
                 mean_pairs=float(_log_int(rng, 1, 500)))
    return c


# ------------------------------------------------------------------ inputs
class Graph:
    """Symmetric CSR with sorted rows; torch device tensors or numpy arrays."""

    def __init__(self, n, row_ptr, col, w):
        self.n, self.row_ptr, self.col, self.w = n, row_ptr, col, w


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _components(n, a, b):
    """Smallest vertex id of each vertex's component."""
    lab = torch.arange(n, device=DEV)
    while True:
        m = lab.clone()
        m.scatter_reduce_(0, b, lab[a], "amin")
        m.scatter_reduce_(0, a, m[b], "amin")
        m = m[m]
        m = m[m]
        if torch.equal(m, lab):
            return lab
        lab = m


def _csr(n, key, gen, wlo, whi):
    """Largest component (ids in order) of the undirected edges a * n + b (a < b,
    unique, sorted), with a weight drawn for every edge."""
    a, b = key // n, key % n
    lab = _components(n, a, b)
    size = torch.bincount(lab, minlength=n)
    keep = lab == torch.argmax(size)
    new = torch.cumsum(keep, 0) - 1
    on = keep[a]
    a, b = new[a[on]], new[b[on]]
    n = int(keep.sum())
    w = torch.randint(wlo, whi + 1, (len(a),), generator=gen, device=DEV)
    order = torch.sort(torch.cat([a * n + b, b * n + a]))
    src = order.values // n
    row = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    col = (order.values % n).to(torch.int32)
    w2 = torch.cat([w, w])[order.indices].to(torch.int32)
    return Graph(n, row, col, w2), keep


def _by_score(score):
    """Rank (larger = more important) by score descending, ties by smaller id."""
    order = torch.sort(score, descending=True, stable=True).indices
    n = len(score)
    rank = torch.empty(n, dtype=torch.int32, device=DEV)
    rank[order] = torch.arange(n - 1, -1, -1, device=DEV, dtype=torch.int32)
    return rank


def _rmat(scale, ef, wmax, gen):
    n, m = 1 << scale, ef << scale
    a = torch.zeros(m, dtype=torch.int64, device=DEV)
    b = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device=DEV)
        down = r >= 0.57 + 0.19
        right = ((r >= 0.57) & ~down) | (r >= 0.57 + 0.19 + 0.19)
        a = 2 * a + down
        b = 2 * b + right
    off = a != b
    key = torch.unique(torch.minimum(a, b)[off] * n + torch.maximum(a, b)[off])
    g, _ = _csr(n, key, gen, 1, wmax)
    return g, _by_score(g.row_ptr[1:] - g.row_ptr[:-1])


def _ba(n, m, wmax, gen):
    """Preferential attachment in linear time (Batagelj and Brandes): edge e of
    vertex e // m ends at the vertex in a uniformly drawn earlier slot."""
    e = torch.arange(n * m, device=DEV)
    p = torch.empty(2 * n * m, dtype=torch.int64, device=DEV)
    p[0::2] = 2 * e
    p[1::2] = (torch.rand(n * m, generator=gen, device=DEV, dtype=torch.float64) * (2 * e + 1)).to(torch.int64)
    while bool((p & 1).any()):
        p = p[p]
    a, b = e // m, p[1::2] // (2 * m)
    off = a != b
    key = torch.unique(torch.minimum(a, b)[off] * n + torch.maximum(a, b)[off])
    g, _ = _csr(n, key, gen, 1, wmax)
    return g, _by_score(g.row_ptr[1:] - g.row_ptr[:-1])


def _grid(side, samples, gen):
    """Grid with a tenth of its edges deleted, weights 500..1500, ranked by the
    number of paths through a vertex in `samples` shortest-path trees."""
    n = side * side
    ids = torch.arange(n, device=DEV).view(side, side)
    key = torch.cat([(ids[:, :-1] * n + ids[:, 1:]).reshape(-1), (ids[:-1] * n + ids[1:]).reshape(-1)])
    drop = torch.rand(len(key), generator=gen, device=DEV)
    key = torch.sort(key[drop.argsort()[len(key) // 10:]]).values
    g, keep = _csr(n, key, gen, 500, 1500)
    # trees from random roots by Bellman-Ford on the grid
    big = 1 << 28
    old = torch.nonzero(keep).view(-1)
    src = torch.repeat_interleave(old, g.row_ptr[1:] - g.row_ptr[:-1])
    dst = old[g.col.long()]
    wr = torch.full((n,), big, dtype=torch.int32, device=DEV)
    wd = wr.clone()
    right, down = dst == src + 1, dst == src + side
    wr[src[right]] = g.w[right]
    wd[src[down]] = g.w[down]
    wr, wd = wr.view(side, side)[:, :-1], wd.view(side, side)[:-1]
    roots = old[torch.randint(0, len(old), (samples,), generator=gen, device=DEV)]
    d = torch.full((samples, n), big, dtype=torch.int32, device=DEV)
    d[torch.arange(samples, device=DEV), roots] = 0
    d = d.view(samples, side, side)
    while True:
        last = d.clone()
        for _ in range(32):
            d[:, :, 1:] = torch.minimum(d[:, :, 1:], d[:, :, :-1] + wr)
            d[:, :, :-1] = torch.minimum(d[:, :, :-1], d[:, :, 1:] + wr)
            d[:, 1:] = torch.minimum(d[:, 1:], d[:, :-1] + wd)
            d[:, :-1] = torch.minimum(d[:, :-1], d[:, 1:] + wd)
        if torch.equal(last, d):
            break
    # parent: the tight neighbour of smallest id (up, left, right, down); the root is its own
    par = ids.expand(samples, side, side).clone()
    at = torch.zeros_like(par, dtype=torch.bool)

    def take(lo, hi, w, by):
        tight = (d[hi] + w == d[lo]) & ~at[lo] & (d[lo] < big)
        par[lo] = torch.where(tight, par_id[lo] + by, par[lo])
        at[lo] |= tight

    par_id = ids.expand(samples, side, side)
    s = slice(None)
    take((s, slice(1, None), s), (s, slice(None, -1), s), wd, -side)
    take((s, s, slice(1, None)), (s, s, slice(None, -1)), wr, -1)
    take((s, s, slice(None, -1)), (s, s, slice(1, None)), wr, 1)
    take((s, slice(None, -1), s), (s, slice(1, None), s), wd, side)
    # descendants by pointer doubling: after k steps, those within 2^k levels
    base = (torch.arange(samples, device=DEV) * (n + 1)).view(-1, 1)
    up = torch.cat([par.view(samples, n), torch.full((samples, 1), n, device=DEV)], 1)
    own = torch.arange(n + 1, device=DEV)
    up = torch.where(up == own, torch.full_like(up, n), up)  # past the root: slot n
    up = (up + base).view(-1)
    cnt = torch.ones(samples * (n + 1), dtype=torch.int64, device=DEV)
    cnt.view(samples, n + 1)[:, n] = 0
    sink = (base + n).view(-1)
    while not bool((up.view(samples, n + 1) == sink.view(-1, 1)).all()):
        cnt = cnt.scatter_add(0, up, cnt)
        cnt[sink] = 0
        up = up[up]
    score = cnt.view(samples, n + 1)[:, :n].sum(0)[old]
    return g, _by_score(score)


def _graph(case, gen):
    if case["family"] == "rmat":
        return _rmat(case["scale"], case["ef"], case["wmax"], gen)
    if case["family"] == "ba":
        return _ba(case["n"], case["m"], case["wmax"], gen)
    return _grid(case["side"], case["samples"], gen)


def _host(g, rank):
    h = Graph(g.n, g.row_ptr.cpu().numpy().view(np.uint64), g.col.cpu().numpy().view(np.uint32),
              g.w.cpu().numpy().view(np.uint32))
    return h, rank.cpu().numpy().view(np.uint32)


def _pairs(g, count, skew, gen):
    """Query pairs: uniform endpoints, or with share `skew` both endpoints drawn by degree."""
    p = torch.randint(0, g.n, (count, 2), generator=gen, device=DEV)
    if skew:
        ends = g.col.long()[torch.randint(0, len(g.col), (count, 2), generator=gen, device=DEV)]
        p = torch.where(torch.rand((count, 1), generator=gen, device=DEV) < skew, ends, p)
    return p.to(torch.int32)


def _buffers(case):
    """The caller's label arrays, allocated once: offsets, hubs, distances (and
    parents), zero past the labels of the graph at hand, whose number varies
    with the seed."""
    ids = (1 << case["scale"]) if case["family"] == "rmat" else case.get("n") or case["side"] ** 2
    n, _, per = _size(case)
    cap = int(2.5 * n * per) + 40 * ids
    return [torch.zeros(ids + 1, dtype=torch.int64, device=DEV)] + [
        torch.zeros(cap, dtype=torch.int32, device=DEV) for _ in range(3 if case.get("parents") else 2)]


def prepare(case, seed):
    gen = _gen(seed)
    g, rank = _graph(case, gen)
    kind = case["kind"]
    if kind == "build":
        opts = {"flags": chl.CHL_FLAG_PARENTS} if case.get("parents") else {}
        s = {"kind": kind, "opts": opts, "host": case.get("host", False), "out": _buffers(case)}
        s["g"], s["rank"] = _host(g, rank) if s["host"] else (g, rank)
        if s["host"]:
            s["out"] = [x.cpu().pin_memory() for x in s["out"]]
        return s
    if kind == "query":
        cuts = [0, 64, 1024, 0]  # hub partitions by rank position
        if case["mode"] == "parts" and g.n > 2048:
            labels = [chl.build_labels(g, rank, root_begin=a, root_end=b) for a, b in zip(cuts, cuts[1:])]
        else:
            labels = [chl.build_labels(g, rank)]
        p = _pairs(g, case["pairs"], case["skew"], gen)
        if case["host"]:
            p = p.cpu().numpy().view(np.uint32)
        return {"kind": kind, "mode": case["mode"], "labels": labels, "pairs": p}
    if kind == "paths":
        labels = chl.build_labels(g, rank, flags=chl.CHL_FLAG_PARENTS)
        return {"kind": kind, "labels": labels, "max_len": case["max_len"],
                "pairs": _pairs(g, case["pairs"], 0.0, gen)}
    g2, rank2 = _ba(case["n2"], 5, 100, gen)
    server = chl.Server()
    sets = [server.add_set(chl.build_labels(g, rank)), server.add_set(chl.build_labels(g2, rank2))]
    rng = np.random.default_rng(case["requests"])  # the sizes belong to the case
    size = rng.geometric(1.0 / max(1.0, case["mean_pairs"]), case["requests"])
    which = rng.integers(0, 2, case["requests"])
    reqs = [(sets[k], _pairs((g, g2)[k], int(c), 0.5, gen).cpu().numpy().view(np.uint32))
            for k, c in zip(which, size)]
    return {"kind": kind, "server": server, "requests": reqs}


# ------------------------------------------------------------------ one pass
def _ok(status):
    if status != chl.CHL_OK:
        raise chl.ChlError(status, chl.chl_last_error())


def run(s):
    kind = s["kind"]
    if kind == "build":
        labels = chl.build_labels(s["g"], s["rank"], **s["opts"])
        out = s["out"]
        if labels.total > len(out[1]):
            raise ValueError("the label buffers of this case are too small")
        mem = chl.CHL_MEM_HOST if s["host"] else chl.CHL_MEM_DEVICE
        stream = torch.cuda.current_stream().cuda_stream
        chl.chl_labels_copy(labels.handle, *(x.data_ptr() for x in out[:3]), mem, stream)
        if s["opts"]:
            _ok(chl.lib().chl_labels_parents(labels.handle, out[3].data_ptr(), mem, stream))
        labels.free()
        return out
    if kind == "query":
        if s["mode"] == "parts":
            return chl.query_partitioned(s["labels"], s["pairs"])
        return s["labels"][0].query(s["pairs"], grouped=s["mode"] == "grouped")
    if kind == "paths":
        p, q = s["pairs"], len(s["pairs"])
        paths = torch.zeros((q, s["max_len"]), dtype=torch.int32, device=DEV)
        lens = torch.empty(q, dtype=torch.int32, device=DEV)
        _ok(chl.lib().chl_path(s["labels"].handle, p.data_ptr(), q, s["max_len"], paths.data_ptr(), lens.data_ptr(),
                               chl.CHL_MEM_DEVICE, torch.cuda.current_stream().cuda_stream))
        return [paths, lens]
    tickets = [s["server"].submit_query(k, p) for k, p in s["requests"]]
    return np.concatenate([s["server"].wait(t)[0] for t in tickets])


# ------------------------------------------------------------------ what a pass cannot do without
def _size(case):
    """(vertices, arcs, labels per vertex) of a case's graph, near enough."""
    if case["family"] == "rmat":
        ids = 1 << case["scale"]
        n, arcs = 0.65 * ids, 1.8 * case["ef"] * ids
    elif case["family"] == "ba":
        n, arcs = case["n"], 2 * case["m"] * case["n"]
    else:
        n, arcs = case["side"] ** 2, 3.6 * case["side"] ** 2
    labels, at, grow = LABELS[case["family"]]
    return n, arcs, labels * (n / at) ** grow


def work(case):
    n, arcs, per = _size(case)
    if case["kind"] == "build":
        width = 12 if case.get("parents") else 8
        return {"bytes": 8 * (n + 1) + 8 * arcs + 4 * n + 8 * (n + 1) + width * per * n, "flops": 0}
    if case["kind"] == "query":
        return {"bytes": case["pairs"] * (12 + 16 * per), "flops": 0}
    if case["kind"] == "paths":
        steps = min(case["max_len"], 0.7 * n ** 0.5 if case["family"] == "grid" else 8)
        return {"bytes": case["pairs"] * (12 + 16 * per + 4 * steps), "flops": 0}
    return {"bytes": case["requests"] * case["mean_pairs"] * (12 + 16 * per), "flops": 0}


def tolerance(case):
    return "exact"


# ------------------------------------------------------------------ the definition, in 64-bit integers
def _all_pairs(g):
    d = torch.full((g.n, g.n), INF, dtype=torch.int64, device=DEV)
    src = torch.repeat_interleave(torch.arange(g.n, device=DEV), g.row_ptr[1:] - g.row_ptr[:-1])
    d[src, g.col.long()] = g.w.long()
    d.fill_diagonal_(0)
    for k in range(g.n):
        d = torch.minimum(d, d[:, k:k + 1] + d[k:k + 1])
    return d


def exact(case, seed):
    """Labels and distances from all-pairs distances: h is a hub of v when it is
    the highest-ranked vertex on the shortest paths between them."""
    if case["kind"] not in ("build", "query"):
        return None
    if case["family"] == "rmat" and case["scale"] > 11 or case.get("n", 0) > 3000 or case.get("side", 0) > 50:
        return None
    gen = _gen(seed)
    g, rank = _graph(case, gen)
    d = _all_pairs(g)
    if case["kind"] == "query":
        p = _pairs(g, case["pairs"], case["skew"], gen).long()
        x = d[p[:, 0], p[:, 1]]
        return torch.where(x < INF, x, torch.full_like(x, 0xFFFFFFFF if case["host"] else -1))
    order = torch.sort(rank, descending=True).indices
    top = torch.full((g.n, g.n), -1, dtype=torch.int64, device=DEV)
    for w in order.tolist():
        on = (top < 0) & (d[:, w:w + 1] + d[w:w + 1] == d) & (d < INF)
        top[on] = w
    by_rank = top[:, order] == order.view(1, -1)  # [v, i]: the i-th hub by rank labels v
    v, i = torch.nonzero(by_rank, as_tuple=True)
    off = torch.zeros(g.n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(by_rank.sum(1), 0)
    out = [x.long() for x in _buffers(case)[:3]]
    for x, y in zip(out, (off, order[i], d[v, order[i]])):
        x[:len(y)] = y
    return out + ([None] if case.get("parents") else [])
