"""Long rows in the pushed levels of the allocation-free assignment, where a block
queues the frontier's rows above 512 entries and spreads them together.  A level
pushes when 64 times its frontier's entries stay below those of the graph, so the
long rows hang off an R-MAT graph of 7.6 M entries.  (A queue holds 256 rows;
more of them in one block's share of a pushed level would take a graph of over a
billion entries.)"""
import functools

import numpy as np
import pytest

import flsynth
import paper_1503_03635_gb300 as fl

LONG, PUSH_DIV = 512, 64


@functools.cache
def _bulk():
    return flsynth.rmat(18, 16, 5)


def _with_hubs(n_hubs, deg):
    """The R-MAT graph and hubs whose `deg` neighbours among its vertices overlap by half."""
    rowp, cols = _bulk()
    n0 = len(rowp) - 1
    hub = np.repeat(np.arange(n0, n0 + n_hubs), deg)
    leaf = (np.arange(n_hubs)[:, None] * (deg // 2) + np.arange(deg)).ravel()
    assert leaf.max() < n0
    src = np.concatenate([np.repeat(np.arange(n0), np.diff(rowp)), hub, leaf])
    dst = np.concatenate([cols, leaf, hub])
    order = np.argsort(src, kind="stable")
    out = np.zeros(n0 + n_hubs + 1, np.int64)
    out[1:] = np.cumsum(np.bincount(src, minlength=n0 + n_hubs))
    return out, dst[order].astype(np.int32), np.arange(n0, n0 + n_hubs)


def _bfs(rowp, cols, opened):
    """Assignment, distances and, per level, (does it push?, long rows in its frontier)."""
    n = len(rowp) - 1
    assign, dist = np.full(n, n, np.int64), np.full(n, -1, np.int32)
    assign[opened], dist[opened] = opened, 0
    level, levels = np.asarray(opened), []
    while len(level):
        deg = rowp[level + 1] - rowp[level]
        levels.append((int(deg.sum()) * PUSH_DIV < len(cols), int((deg > LONG).sum())))
        at = np.repeat(rowp[level] - (np.cumsum(deg) - deg), deg) + np.arange(deg.sum())
        u, lab = cols[at], np.repeat(assign[level], deg)
        new = dist[u] < 0
        u, lab = u[new], lab[new]
        np.minimum.at(assign, u, lab)
        level = np.unique(u)
        dist[level] = len(levels)
    return np.where(dist < 0, -1, assign).astype(np.int32), dist, levels


# rows at the limit of the queue, one row of several turns of the block, rows for
# one warp of each of 32 in a block (the first 32 of the frontier), for five blocks
@pytest.mark.gpu
@pytest.mark.parametrize("n_hubs,deg", [(2, 512), (2, 513), (1, 3000), (1, 20_000), (32, 520), (40, 600), (150, 600)])
def test_long_rows_are_pushed(n_hubs, deg):
    import torch
    rowp, cols, hubs = _with_hubs(n_hubs, deg)
    want_a, want_d, levels = _bfs(rowp, cols, hubs)
    assert levels[0] == (True, n_hubs if deg > LONG else 0)
    n = len(rowp) - 1
    is_open = np.zeros(n, np.uint8)
    is_open[hubs] = 1
    to = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    a = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    d = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    fl.assign_nearest_noalloc(to(rowp), to(cols), to(is_open), a, d)
    assert np.array_equal(d.cpu().numpy(), want_d)
    assert np.array_equal(a.cpu().numpy(), want_a)
