"""The resident BFS of the assignment on graphs whose levels push and pull in turn:
rows at the length that a block's warps share, thin frontiers after wide ones (which
are listed first) and wide ones after thin ones, several labels at one vertex,
sources without edges and unreached parts."""
import numpy as np
import pytest

import flsynth
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _csr(n, a, b):
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    rowp = np.zeros(n + 1, np.int64)
    rowp[1:] = np.cumsum(np.bincount(src, minlength=n))
    return rowp, dst[np.argsort(src, kind="stable")].astype(np.int32)


def _bfs(rowp, cols, opened):
    n = len(rowp) - 1
    assign, dist = np.full(n, n, np.int64), np.full(n, -1, np.int32)
    assign[opened], dist[opened] = opened, 0
    level, at = np.asarray(opened), 0
    while len(level):
        at += 1
        deg = rowp[level + 1] - rowp[level]
        e = np.repeat(rowp[level] - (np.cumsum(deg) - deg), deg) + np.arange(deg.sum())
        u, lab = cols[e], np.repeat(assign[level], deg)
        new = dist[u] < 0
        np.minimum.at(assign, u[new], lab[new])
        level = np.unique(u[new])
        dist[level] = at
    return np.where(dist < 0, -1, assign).astype(np.int32), dist


def _grid(w, h):
    v = np.arange(w * h).reshape(h, w)
    return _csr(w * h, np.concatenate([v[:, :-1].ravel(), v[:-1].ravel()]),
                np.concatenate([v[:, 1:].ravel(), v[1:].ravel()]))


def _bulk_and(extra_n, a, b):
    """An R-MAT graph of 2^17 vertices with `extra_n` more and the given edges."""
    rowp, cols = flsynth.rmat(17, 8, 11)
    n0 = len(rowp) - 1
    src = np.repeat(np.arange(n0), np.diff(rowp))
    keep = src < cols
    return (*_csr(n0 + extra_n, np.concatenate([src[keep], a]), np.concatenate([cols[keep], b])), n0)


def _case(name):
    if name == "grid":                      # thin throughout; 700 levels
        rowp, cols = _grid(401, 301)
        return rowp, cols, [5, 60_000]
    if name == "large grid":                # above the size from which a pulled level is listed
        rowp, cols = _grid(801, 601)
        return rowp, cols, list(range(0, 801 * 601, 40_009))
    if name == "wide then thin":            # half of a large graph open, a long path hanging off it
        n0, tail = 1 << 19, 3_000
        rng = np.random.default_rng(3)
        a, b = rng.integers(0, n0, n0), rng.integers(0, n0, n0)
        rowp, cols = _csr(n0 + tail, np.concatenate([a[a != b], np.arange(n0 - 1, n0 + tail - 1)]),
                          np.concatenate([b[a != b], np.arange(n0, n0 + tail)]))
        return rowp, cols, list(range(0, n0, 2))
    if name == "hubs":                      # two thin levels, then hubs of 100,000 entries (pulled)
        rowp, cols = _csr(100_050, np.repeat(np.arange(50), 100_000), np.tile(50 + np.arange(100_000), 50))
        return rowp, cols, [77, 50_123]
    if name.startswith("row"):              # pushed rows, overlapping by half
        deg, hubs = int(name[3:]), 3
        n0 = 1 << 17
        leaf = (np.arange(hubs)[:, None] * (deg // 2) + np.arange(deg)).ravel()
        rowp, cols, n0 = _bulk_and(hubs, np.repeat(n0 + np.arange(hubs), deg), leaf)
        return rowp, cols, [n0, n0 + 1, n0 + 2]
    if name == "many":                      # 40 rows of 100 entries in one block's share, some vertices with 20 offers
        n0, hubs = 1 << 17, 40
        leaf = (np.arange(hubs)[:, None] * 5 + np.arange(100)).ravel()
        rowp, cols, n0 = _bulk_and(hubs, np.repeat(n0 + np.arange(hubs), 100), leaf)
        return rowp, cols, list(range(n0, n0 + hubs))
    rowp, cols, n0 = _bulk_and(100, np.zeros(0, np.int64), np.zeros(0, np.int64))
    return rowp, cols, [3, n0 + 7, n0 + 50]  # "isolated": sources without edges, unreached vertices


@pytest.mark.parametrize("name", ["grid", "large grid", "wide then thin", "hubs", "row63", "row64", "row65",
                                  "row128", "row129", "row4097", "many", "isolated"])
def test_assignment_matches_plain_bfs(name):
    rowp, cols, opened = _case(name)
    n = len(rowp) - 1
    want_a, want_d = _bfs(rowp, cols, opened)
    cost = np.full(n, np.inf)
    cost[opened] = 0.5  # balls of radius 0: every facility opens
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    s = fl.Solve(g)
    s.compute_radii(cost, np.ones(n, np.uint8))
    _, n_open = s.open_facilities()
    assert n_open == len(opened)
    g.profile(True)
    g.profile_reset()
    a, d = s.assign_clients()
    assert g.profile_query("bfs")["launches"] == 1  # the resident kernel
    assert np.array_equal(d, want_d) and np.array_equal(a, want_a)
    s.close()
    g.close()


def test_a_few_sources_beside_hubs_do_not_read_every_row():
    # with a pull at every level the assignment took 2.4 times the host-driven rounds
    rowp, cols, _ = _case("hubs")
    n = len(rowp) - 1
    cost = np.full(n, np.inf)
    cost[77] = 0.5
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    s = fl.Solve(g)
    s.compute_radii(cost, np.ones(n, np.uint8))
    s.open_facilities()
    g.profile(True)
    ms = {}
    for dense_div in (8, 9):  # 9: host-driven
        g.set_schedule(dense_div=dense_div)
        ms[dense_div] = []
        for _ in range(6):
            g.profile_reset()
            s.assign_clients()
            ms[dense_div].append(g.profile_query("bfs")["ms"])
    assert min(ms[8]) < 1.5 * min(ms[9]), ms
    s.close()
    g.close()
