"""What is measured: the facility-location path through its public entry points.

A case names a family of work (``kind``) and its sizes.  Graphs are the two
families that the repository's workloads use, R-MAT (0.57, 0.19, 0.19, 0.05) and
Erdos-Renyi, symmetrised and deduplicated, with any number of vertices (odd ones
among them); costs are uniform constants or log-uniform, client and facility sets
are random subsets.  ``listed()`` says what each case stands for.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1503_03635_gb300 as fl

DEV = "cuda"
RMAT = (0.57, 0.19, 0.19)


def listed():
    return [
        # the smallest ordinary call: one instance on a 10^4-vertex random graph, sketches included,
        # where every vertex is a client and a facility at cost 20; latency and launches count
        dict(name="solve_er10k", kind="solve", graph="er", n=10_000, ef=4.0, k=16, clients=1.0, facs=1.0, lo=20.0, hi=20.0),
        # an ordinary social-graph solve: 2^20 vertices, all of them clients and facilities, k = 32
        dict(name="solve_rmat20", kind="solve", graph="rmat", n=1 << 20, ef=16.0, k=32, clients=1.0, facs=1.0, lo=5.0, hi=500.0),
        # the largest: half the vertices clients, a tenth facilities, costs over three decades, k = 16
        # (a size of which three states fit the card; the graph no longer fits L2 by a factor of fifteen)
        dict(name="solve_rmat24", kind="solve", graph="rmat", n=1 << 24, ef=16.0, k=16, clients=0.5, facs=0.1, lo=10.0, hi=1e4),
        # a script's one call on host arrays: graph creation, sketches and every phase, results on the host
        dict(name="oneshot_rmat16", kind="oneshot", graph="rmat", n=61_001, ef=16.0, k=16, clients=0.6, facs=0.5, lo=5.0, hi=200.0),
        # one query on a resident graph with built sketches: a client subset and one opening cost
        dict(name="query_rmat22", kind="query", graph="rmat", n=(1 << 22) - 77, ef=16.0, k=32, clients=0.02, facs=1.0, lo=100.0, hi=100.0),
        # many small independent graphs solved in one call
        dict(name="batch_er64", kind="union", parts=64, n_lo=1000, n_hi=50_000, ef=5.0, k=32, clients=1.0, facs=1.0, lo=5.0, hi=500.0),
        # many instances (own client sets and costs) on one resident graph in one call
        dict(name="batch_rmat18", kind="replicas", graph="rmat", n=1 << 18, ef=16.0, k=32, inst=16, clients=0.2, facs=1.0, lo=5.0, hi=500.0),
        # road-like use: integer edge lengths in [1, 100], sketches in distance order, MIS and assignment by length
        dict(name="weighted_rmat16", kind="weighted", graph="rmat", n=65_536, ef=16.0, k=16, max_len=100, clients=1.0, facs=1.0, lo=5.0, hi=500.0),
        # the accuracy study: exact ball sizes of sampled vertices and their sketch estimates, distances 0..20
        dict(name="accuracy_rmat18", kind="accuracy", graph="rmat", n=1 << 18, ef=16.0, k=16, sources=1000, dist=20, clients=0.5),
        # radii from exact client counts (a BFS per facility) in place of the estimates
        dict(name="exact_radii_rmat16", kind="exact_radii", graph="rmat", n=65_536, ef=16.0, k=16, clients=0.5, facs=0.05, lo=5.0, hi=500.0),
        # the paper's own opening phase with eps > 0 on a resident graph with built sketches
        dict(name="eps_rmat16", kind="eps", graph="rmat", n=65_536, ef=16.0, k=16, eps=0.1, clients=1.0, facs=1.0, lo=5.0, hi=500.0),
        # a latency-critical loop that may not allocate: nearest open facility for a given open set
        dict(name="assign_rmat19", kind="assign", graph="rmat", n=500_009, ef=16.0, k=0, facs=0.01),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "oneshot", "query", "union", "replicas", "weighted", "accuracy",
                       "exact_radii", "eps", "assign"])
    cost = rng.choice([(20.0, 20.0), (5.0, 500.0), (10.0, 1e4)])
    c = dict(kind=kind, graph=rng.choice(["rmat", "rmat", "er"]), ef=float(rng.choice([4, 8, 16])),
             k=rng.choice([4, 8, 16, 24, 32]), clients=rng.choice([1.0, 0.5, 0.1]), facs=rng.choice([1.0, 0.5, 0.1]),
             lo=cost[0], hi=cost[1])
    if kind == "solve":
        return dict(c, n=_log_int(rng, 1_000, 5_000_000))
    if kind == "oneshot":
        return dict(c, n=_log_int(rng, 1_000, 300_000))
    if kind == "query":
        u = math.exp(rng.uniform(math.log(10.0), math.log(1000.0)))
        return dict(c, n=_log_int(rng, 30_000, 4_000_000), facs=1.0, clients=rng.choice([0.5, 0.1, 0.01]), lo=u, hi=u)
    if kind == "union":
        hi = _log_int(rng, 2_000, 50_000)
        return dict(kind=kind, parts=rng.randint(3, 64), n_lo=min(hi, _log_int(rng, 100, 5_000)), n_hi=hi,
                    ef=rng.choice([2.0, 4.0, 8.0]), k=c["k"], clients=c["clients"], facs=c["facs"], lo=c["lo"], hi=c["hi"])
    if kind == "replicas":
        return dict(c, n=_log_int(rng, 5_000, 260_000), inst=rng.randint(2, 16), clients=rng.choice([0.5, 0.1, 0.02]),
                    facs=1.0)
    if kind == "weighted":
        return dict(c, n=_log_int(rng, 1_000, 65_000), k=rng.choice([4, 8, 16]), max_len=rng.choice([1, 10, 100]))
    if kind == "accuracy":
        return dict(kind=kind, graph=c["graph"], n=_log_int(rng, 5_000, 260_000), ef=c["ef"], k=c["k"],
                    sources=rng.randint(10, 1000), dist=rng.randint(3, 20), clients=c["clients"])
    if kind == "exact_radii":
        return dict(c, n=_log_int(rng, 2_000, 65_000), facs=rng.choice([0.05, 0.01]))
    if kind == "eps":
        return dict(c, n=_log_int(rng, 1_000, 65_000), eps=rng.choice([0.1, 0.3, 1.0]), lo=5.0, hi=500.0)
    return dict(kind="assign", graph=c["graph"], n=_log_int(rng, 5_000, 1_000_000), ef=c["ef"], k=0,
                facs=rng.choice([0.1, 0.01, 0.001]))


# ------------------------------------------------------------------ inputs


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _csr(n, src, dst):
    """Symmetric, deduplicated CSR without self-loops of the given draws."""
    key = torch.cat([src.long() * n + dst, dst.long() * n + src])
    key = key[src.repeat(2) != dst.repeat(2)]
    key = torch.unique(key)
    rows = torch.div(key, n, rounding_mode="floor")
    cols = (key - rows * n).int()
    rowp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rowp, cols.contiguous()


def _graph(kind, n, ef, gen):
    m = int(ef * n)
    if kind == "er":
        return _csr(n, torch.randint(n, (m,), generator=gen, device=DEV, dtype=torch.int32),
                    torch.randint(n, (m,), generator=gen, device=DEV, dtype=torch.int32))
    bits = max(1, (n - 1).bit_length())
    src = torch.zeros(m, dtype=torch.int32, device=DEV)
    dst = torch.zeros(m, dtype=torch.int32, device=DEV)
    a, b, c = RMAT
    for _ in range(bits):
        r = torch.rand(m, generator=gen, device=DEV)
        low = r >= a + b
        right = ((r >= a) & (r < a + b)) | (r >= a + b + c)
        src = src * 2 + low
        dst = dst * 2 + right
    # a random numbering of the 2^bits ids; edges with an end at or above n fall out
    perm = torch.randperm(1 << bits, generator=gen, device=DEV, dtype=torch.int32)
    src, dst = perm[src.long()], perm[dst.long()]
    if n < 1 << bits:
        keep = (src < n) & (dst < n)
        src, dst = src[keep], dst[keep]
    return _csr(n, src, dst)


def _subset(n, p, gen):
    if p >= 1.0:
        return torch.ones(n, dtype=torch.uint8, device=DEV)
    m = (torch.rand(n, generator=gen, device=DEV) < p).to(torch.uint8)
    m[torch.randint(n, (1,), generator=gen, device=DEV)] = 1
    return m


def _costs(n, lo, hi, facs, gen):
    """Opening costs: one constant, or log-uniform in [lo, hi]; +inf where not a facility."""
    u = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    cost = torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo))) if hi > lo else torch.full_like(u, lo)
    return torch.where(_subset(n, facs, gen) > 0, cost, torch.full_like(cost, math.inf))


def _lengths(rowp, cols, max_len, seed):
    """Integer lengths in [1, max_len], the same for both directions of an edge (a hash of the unordered pair)."""
    n = len(rowp) - 1
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rowp[1:] - rowp[:-1])
    a, b = torch.minimum(src, cols.long()), torch.maximum(src, cols.long())
    x = (a * 1_000_003 + b * 7_368_787 + seed * 97 + 12345) & 0x7FFFFFFF
    x = (x ^ (x >> 15)) * 739_982_445 & 0x7FFFFFFF
    x = (x ^ (x >> 12)) * 695_872_825 & 0x7FFFFFFF
    x = x ^ (x >> 15)
    return (x % max_len + 1).int()


def _part_sizes(case):
    """Log-uniformly spread sizes, the same for every seed."""
    u = (np.arange(case["parts"]) * 0.618033988749895 + 0.5) % 1.0
    return np.exp(math.log(case["n_lo"]) + u * (math.log(case["n_hi"]) - math.log(case["n_lo"]))).astype(np.int64)


def _inputs(case, seed):
    """Everything that the seed gives: the same for prepare() and exact()."""
    gen = _generator(seed)
    d = dict(rank_seed=1 + int(seed))
    if case["kind"] == "union":
        n_of = _part_sizes(case)
        parts = [_graph("er", int(m), case["ef"], gen) for m in n_of]
        n = int(n_of.sum())
        d.update(n_of=n_of, parts=parts)
        per = _costs(len(n_of), case["lo"], case["hi"], 1.0, gen)
        cost = per[torch.repeat_interleave(torch.arange(len(n_of), device=DEV), torch.from_numpy(n_of).to(DEV))]
        fac = _subset(n, case["facs"], gen)
        d.update(cost=torch.where(fac > 0, cost, torch.full_like(cost, math.inf)), client=_subset(n, case["clients"], gen))
        return d
    n = case["n"]
    d["rowp"], d["cols"] = _graph(case["graph"], n, case["ef"], gen)
    if case["kind"] == "assign":
        d["open"] = _subset(n, case["facs"], gen)
    elif case["kind"] == "accuracy":
        d["src"] = torch.randint(n, (case["sources"],), generator=gen, device=DEV, dtype=torch.int32)
        d["pred"] = _subset(n, case["clients"], gen)
    elif case["kind"] == "replicas":
        d["cost"] = torch.cat([torch.full((n,), float(c), dtype=torch.float64, device=DEV)
                               for c in _costs(case["inst"], case["lo"], case["hi"], 1.0, gen)])
        d["client"] = torch.cat([_subset(n, case["clients"], gen) for _ in range(case["inst"])])
    else:
        d["cost"] = _costs(n, case["lo"], case["hi"], case["facs"], gen)
        d["client"] = _subset(n, case["clients"], gen)
        if case["kind"] == "weighted":
            d["len"] = _lengths(d["rowp"], d["cols"], case["max_len"], int(seed))
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    s = dict(kind=kind, k=case["k"], seed=d["rank_seed"], case=case)
    n = int(sum(d["n_of"])) if kind == "union" else case["n"]
    if kind == "oneshot":
        s.update({a: d[a].cpu().numpy() for a in ("rowp", "cols", "cost", "client")})
        return s
    s.update({a: d[a] for a in ("rowp", "cols", "cost", "client", "open", "src", "pred") if a in d})
    total = n * case.get("inst", 1)
    if kind == "accuracy":
        shape = (case["sources"], case["dist"] + 1)
        s.update(sizes=torch.empty(shape, dtype=torch.int64, device=DEV),
                 est=torch.empty(shape, dtype=torch.float64, device=DEV))
    else:
        s.update(open_out=torch.empty(total, dtype=torch.uint8, device=DEV),
                 assign=torch.empty(total, dtype=torch.int32, device=DEV),
                 dist=torch.empty(total, dtype=torch.int32, device=DEV),
                 radii=torch.empty(total, dtype=torch.float64, device=DEV))
    if kind == "eps":
        s.update(fac_iter=torch.empty(n, dtype=torch.int32, device=DEV),
                 cli_iter=torch.empty(n, dtype=torch.int32, device=DEV))
    torch.cuda.empty_cache()  # the library allocates beside torch's cache
    if kind == "union":
        s["batch"] = fl.Batch.union(d["parts"])
        return s
    if kind == "assign":
        return s
    s["graph"] = fl.Graph(s["rowp"], s["cols"], lengths=d.get("len"))
    if kind in ("query", "replicas", "accuracy", "exact_radii", "eps"):
        s["graph"].build_sketches(s["k"], s["seed"])
    if kind in ("query", "exact_radii", "eps"):
        s["solve"] = fl.Solve(s["graph"])
    if kind == "replicas":
        s["batch"] = fl.Batch.replicas(s["graph"], case["inst"])
    return s


# ------------------------------------------------------------------ one pass


def _phases(s, solve, radii):
    """Facilities, assignment and objective after the radii."""
    _, n_open = solve.open_facilities(s["open_out"])
    solve.assign_clients(s["assign"], s["dist"])
    obj, dist_sum, unserved = solve.objective()
    out = dict(open=s["open_out"], assign=s["assign"], dist=s["dist"], n_open=n_open, objective=obj,
               dist_sum=dist_sum, unserved=unserved)
    return dict(out, radii=radii) if radii is not None else out


def run(s):
    kind = s["kind"]
    if kind in ("solve", "weighted"):
        g = s["graph"]
        g.build_sketches(s["k"], s["seed"])
        solve = fl.Solve(g)
        solve.compute_radii(s["cost"], s["client"], s["radii"])
        out = _phases(s, solve, s["radii"])
        solve.close()
        return dict(out, stats=g.stats())
    if kind == "oneshot":
        r = fl.solve(s["rowp"], s["cols"], s["k"], s["seed"], s["cost"], s["client"])
        r["solve"].close()
        r["graph"].close()
        return {a: r[a] for a in ("open", "assign", "dist", "n_open", "objective", "dist_sum", "radii", "stats")}
    if kind == "query":
        s["solve"].compute_radii(s["cost"], s["client"], s["radii"])
        return _phases(s, s["solve"], s["radii"])
    if kind in ("union", "replicas"):
        return s["batch"].solve(s["k"], s["seed"], s["cost"], s["client"], s["open_out"], s["assign"], s["dist"])
    if kind == "accuracy":
        s["graph"].ball_sizes(s["src"], s["case"]["dist"], s["pred"], s["sizes"])
        s["graph"].ball_estimates(s["src"], s["case"]["dist"], s["pred"], s["est"])
        return dict(sizes=s["sizes"], estimates=s["est"])
    if kind == "exact_radii":
        s["solve"].compute_radii_exact(s["cost"], s["client"], s["radii"])
        return _phases(s, s["solve"], s["radii"])
    if kind == "eps":
        s["solve"].open_facilities_eps(s["case"]["eps"], s["cost"], s["client"], s["open_out"], s["fac_iter"],
                                       s["cli_iter"])
        s["solve"].assign_clients(s["assign"], s["dist"])
        obj, dist_sum, unserved = s["solve"].objective()
        return dict(open=s["open_out"], assign=s["assign"], dist=s["dist"], fac_iter=s["fac_iter"],
                    cli_iter=s["cli_iter"], objective=obj, dist_sum=dist_sum, unserved=unserved)
    fl.assign_nearest_noalloc(s["rowp"], s["cols"], s["open"], s["assign"], s["dist"])
    return dict(assign=s["assign"], dist=s["dist"])


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    """Bytes: the CSR (about 2 x draws entries of 4 B, 8 B per row), costs and
    masks read once, per-vertex results (radius, open flag, assignment, distance)
    written once.  No case needs floating-point work to speak of."""
    n = int(_part_sizes(case).sum()) if case["kind"] == "union" else case["n"]
    graph = 8 * n + 4 * 2 * case["ef"] * n
    if case["kind"] == "assign":
        return dict(bytes=graph + 9 * n, flops=0)
    if case["kind"] == "accuracy":
        return dict(bytes=graph + n + case["sources"] * (4 + 16 * (case["dist"] + 1)), flops=0)
    if case["kind"] == "weighted":
        graph += 4 * 2 * case["ef"] * n
    return dict(bytes=graph + 26 * n * case.get("inst", 1), flops=0)


def tolerance(case):
    """Ids, distances, masks and counts are exact.  Radii are a fixed sequence of
    64-bit operations; estimates and the objective are 64-bit sums, whose order
    may differ (2^-53 per operation, at most some thousands of operations deep)."""
    if case["kind"] == "assign":
        return "exact"
    return {"rel": 1e-12, "max": 1e-12, "differ": 0.0}


# ------------------------------------------------------------------ 64-bit reference
# The definitions in plain torch: sketches as the k smallest hashes within h hops,
# HIP weights, the radius of Eq. 1, the lexicographically-first MIS by (radius,
# priority) and the nearest open facility.


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _hashes(state, ids):
    with np.errstate(over="ignore"):
        return _mix(np.uint64(state) + (ids.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))


def _priority_state(seed):
    with np.errstate(over="ignore"):
        return int(_mix(np.array([seed], np.uint64) + np.uint64(0x9E3779B97F4A7C15))[0])


def _sketch_groups(rowp, cols, rank, k):
    """Per hop: (vertex, id) of the entries gained and, per vertex that gained,
    nothing else is needed but the sketch size and its k-th hash.  Yields
    (hop, v, u, counted, weight) per entry."""
    n = len(rowp) - 1
    order = np.argsort(rank, kind="stable")
    ordinal = np.empty(n, np.int64)
    ordinal[order] = np.arange(n)
    vertex_of = torch.from_numpy(order).to(DEV)
    value_of = torch.from_numpy(rank[order].astype(np.float64)).to(DEV)
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rowp[1:] - rowp[:-1])
    dst = cols.long()
    sketch = torch.arange(n, device=DEV) * n + torch.from_numpy(ordinal).to(DEV)  # keys vertex * n + ordinal
    delta = sketch
    hop = 0
    while True:
        v, o = torch.div(delta, n, rounding_mode="floor"), delta % n
        owner = torch.div(sketch, n, rounding_mode="floor")
        start = torch.searchsorted(owner, torch.arange(n + 1, device=DEV))
        size = start[1:] - start[:-1]
        full = size == k
        kth = torch.where(full, (start[:-1] + k - 1).clamp(max=len(sketch) - 1), torch.zeros_like(size))
        kth = sketch[kth] % n
        weight = torch.where(full, 18446744073709551616.0 / value_of[kth], torch.ones(n, dtype=torch.float64, device=DEV))
        counted = ~(full[v] & (o == kth[v]))
        yield hop, v, vertex_of[o], counted, weight
        first = torch.searchsorted(v, torch.arange(n + 1, device=DEV))
        cnt = (first[1:] - first[:-1])[dst]  # entries that cross each edge
        at = torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
        j = torch.arange(int(cnt.sum()), device=DEV) - at + torch.repeat_interleave(first[:-1][dst], cnt)
        cand = torch.repeat_interleave(src, cnt) * n + o[j]
        both = torch.unique(torch.cat([sketch, cand]))
        owner = torch.div(both, n, rounding_mode="floor")
        start = torch.searchsorted(owner, torch.arange(n + 1, device=DEV))
        new = both[torch.arange(len(both), device=DEV) - start[owner] < k]
        at = torch.searchsorted(sketch, new).clamp(max=len(sketch) - 1)
        delta = new[sketch[at] != new]
        sketch = new
        hop += 1
        if len(delta) == 0:
            return


def _radius_walk(per_hop, last, cost):
    """Root of sum_h W_h max(0, r - h) = cost; per_hop: W_h for h = 0.. and `last`, each vertex's last distance."""
    N = torch.zeros_like(cost)
    G = torch.zeros_like(cost)
    r = torch.full_like(cost, math.inf)
    todo = cost < math.inf
    for j, w in enumerate(per_hop):
        N = torch.where(todo, N + w, N)
        end = todo & (last == j)
        r = torch.where(end & (N > 0), j + (cost - G) / N, r)
        todo = todo & ~end
        nxt = G + N
        hit = todo & (nxt >= cost)
        r = torch.where(hit, j + (cost - G) / N, r)
        todo = todo & ~hit
        G = torch.where(todo, nxt, G)
    return r


def _spread(x, src, dst):
    """Each vertex's smallest value among its neighbours' and its own."""
    return x.scatter_reduce(0, src, x[dst], "amin", include_self=True)


def _select(rowp, cols, radii, client, prio, far):
    """Open set: lexicographically-first MIS of the graph that joins facilities whose balls share a client."""
    n = len(rowp) - 1
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rowp[1:] - rowp[:-1])
    dst = cols.long()
    cand = (radii < math.inf).nonzero().flatten().cpu().numpy()
    order = cand[np.lexsort((prio[cand], radii.cpu().numpy()[cand]))]
    key = torch.full((n,), -1, dtype=torch.int64, device=DEV)
    key[torch.from_numpy(order).to(DEV)] = torch.arange(len(order), device=DEV)
    ball = torch.where(radii < math.inf, torch.floor(radii).clamp(max=float(far)), torch.zeros_like(radii)).long()
    state = torch.where(key >= 0, 0, 2)
    big = n + 5
    claimed = torch.zeros(n, dtype=torch.bool, device=DEV)
    while bool((state == 0).any()):
        T = int(ball[state == 0].max())
        cov = torch.full((n,), big, dtype=torch.int64, device=DEV)
        for t in range(T + 1):
            cov = torch.where((state == 0) & (ball == T - t), torch.minimum(cov, key), cov)
            if t < T:
                cov = _spread(cov, src, dst)
        x = torch.where((client > 0) & (cov < big), torch.where(claimed, torch.zeros_like(cov), cov + 1),
                        torch.full_like(cov, big))
        joins = torch.zeros(n, dtype=torch.bool, device=DEV)
        dies = torch.zeros_like(joins)
        for b in range(T + 1):
            mine = (state == 0) & (ball == b)
            dies |= mine & (x == 0)
            joins |= mine & (x == key + 1)
            if b < T:
                x = _spread(x, src, dst)
        state = torch.where(dies, 2, torch.where(joins, 1, state))
        won = torch.zeros(big + 1, dtype=torch.bool, device=DEV)
        won[key[joins]] = True
        claimed |= (client > 0) & won[cov]
    return state == 1


def _nearest(rowp, cols, is_open, label):
    n = len(rowp) - 1
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rowp[1:] - rowp[:-1])
    dst = cols.long()
    big = 1 << 40
    best = torch.where(is_open, label, torch.full_like(label, big))
    dist = torch.where(is_open, 0, -1)
    for level in range(1, n + 1):
        new = _spread(best, src, dst)
        fresh = (dist < 0) & (new < big)
        if not bool(fresh.any()):
            break
        best = torch.where(fresh, new, best)
        dist = torch.where(fresh, level, dist)
    return torch.where(best < big, best, torch.full_like(best, -1)).int(), dist.int()


def _sketch_radii(rowp, cols, rank, k, cost, client):
    """(radii, largest distance any ball can need)."""
    n = len(rowp) - 1
    per_hop, root = [], torch.zeros(n, dtype=torch.int64, device=DEV)
    last = torch.zeros(n, dtype=torch.int64, device=DEV)
    for hop, v, u, counted, weight in _sketch_groups(rowp, cols, rank, k):
        hits = torch.zeros(n, dtype=torch.float64, device=DEV)
        hits.index_add_(0, v, (counted & (client[u] > 0)).double())
        per_hop.append(hits * weight)
        last[v] = hop
        root = torch.maximum(root, last)
    return _radius_walk(per_hop, last, cost), 2 * int(root.max()) + n.bit_length()


def _finish(rowp, cols, radii, cost, client, prio, label, far):
    is_open = _select(rowp, cols, radii, client, prio, far)
    assign, dist = _nearest(rowp, cols, is_open, label)
    return is_open, assign, dist


def _objective(is_open, cost, client, dist):
    served = (client > 0) & (dist >= 0)
    return float(cost[is_open].sum()) + float(dist[served].sum())


def exact(case, seed):
    kind, k = case["kind"], case["k"]
    if kind in ("weighted", "eps", "assign"):
        return None  # a Dijkstra per vertex, and the iterations' decisions: over the time; no floating outputs
    if kind == "union":
        entries = int(_part_sizes(case).sum()) * case["ef"] * 2 * k
    else:
        entries = case["n"] * case["ef"] * 2 * k
    if entries > 6e8:
        return None  # a hop's candidates (one per entry of every neighbour's sketch) are sorted as a whole
    d = _inputs(case, seed)
    if kind == "union":
        base = np.concatenate([[0], np.cumsum(d["n_of"])])
        local = np.concatenate([np.arange(m) for m in d["n_of"]])
        edges = np.cumsum([0] + [len(c) for _, c in d["parts"]])
        rowp = torch.cat([r[:-1] + int(e) for (r, _), e in zip(d["parts"], edges)] +
                         [torch.tensor([int(edges[-1])], device=DEV)])
        cols = torch.cat([c.long() + int(b) for (_, c), b in zip(d["parts"], base)])
    else:
        rowp, cols = d["rowp"], d["cols"]
        local = np.arange(case["n"])
    rank, prio = _hashes(d["rank_seed"], local), _hashes(_priority_state(d["rank_seed"]), local)
    if kind == "accuracy":
        pred, src, D = d["pred"], d["src"].long(), case["dist"]
        est = torch.zeros((len(src), D + 1), dtype=torch.float64, device=DEV)
        run_sum = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        done = 0
        for hop, v, u, counted, weight in _sketch_groups(rowp, cols, rank, k):
            if hop > D:
                break
            hits = torch.zeros_like(run_sum).index_add_(0, v, (counted & (pred[u] > 0)).double())
            run_sum = run_sum + hits * weight
            est[:, hop] = run_sum[src]
            done = hop
        est[:, done + 1:] = run_sum[src][:, None]
        return dict(sizes=None, estimates=est)
    label = torch.from_numpy(local).to(DEV)
    if kind == "replicas":
        outs = []
        for i in range(case["inst"]):
            part = slice(i * case["n"], (i + 1) * case["n"])
            cost, client = d["cost"][part], d["client"][part]
            radii, far = _sketch_radii(rowp, cols, rank, k, cost, client)
            is_open, _, dist = _finish(rowp, cols, radii, cost, client, prio, label, far)
            outs.append(_objective(is_open, cost, client, dist))
        return dict(objective=np.array(outs))
    cost, client = d["cost"], d["client"]
    if kind == "exact_radii":
        radii, far = _exact_count_radii(rowp, cols, cost, client)
    else:
        radii, far = _sketch_radii(rowp, cols, rank, k, cost, client)
    is_open, assign, dist = _finish(rowp, cols, radii, cost, client, prio, label, far)
    if kind == "union":
        return dict(objective=np.array([_objective(is_open[a:b], cost[a:b], client[a:b], dist[a:b])
                                        for a, b in zip(base[:-1], base[1:])]))
    return dict(radii=radii, objective=_objective(is_open, cost, client, dist))


def _exact_count_radii(rowp, cols, cost, client):
    """Radii with W_h = the number of clients at distance exactly h, by one dense BFS per block of facilities."""
    n = len(rowp) - 1
    adj = torch.sparse_csr_tensor(rowp, cols.long(), torch.ones(len(cols), device=DEV), size=(n, n))
    radii = torch.full((n,), math.inf, dtype=torch.float64, device=DEV)
    facs = (cost < math.inf).nonzero().flatten()
    far = 0
    for part in facs.split(512):
        front = torch.zeros((n, len(part)), device=DEV)
        front[part, torch.arange(len(part), device=DEV)] = 1.0
        seen = front > 0
        per_hop, last, hop = [], torch.zeros(len(part), dtype=torch.int64, device=DEV), 0
        while bool((front > 0).any()):
            per_hop.append((front.double() * client.double()[:, None]).sum(0))
            last = torch.where((front > 0).any(0), hop, last)
            new = ((adj @ front) > 0) & ~seen
            seen |= new
            front = new.float()
            hop += 1
        far = max(far, int(last.max()))
        radii[part] = _radius_walk(per_hop, last, cost[part])
    return radii, 2 * far + 2
