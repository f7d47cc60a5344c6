"""Exact ball sizes on rows that are cut into work items: the bits that a row needs
come with its first item, with its last, or with several."""
import numpy as np
import pytest

import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _csr(n, a, b):
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    rowp = np.zeros(n + 1, np.int64)
    rowp[1:] = np.cumsum(np.bincount(src, minlength=n))
    order = np.lexsort((dst, src))
    return rowp, dst[order].astype(np.int32)


def _sizes(rowp, cols, src, D, pred):
    out = np.zeros((len(src), D + 1), np.int64)
    for i, s in enumerate(src):
        dist = np.full(len(rowp) - 1, -1)
        dist[s], level = 0, [s]
        for h in range(D + 1):
            nxt = np.unique(np.concatenate([cols[rowp[v]:rowp[v + 1]] for v in level])) if len(level) else []
            out[i, h] = pred[(dist >= 0) & (dist <= h)].sum()
            level = [u for u in nxt if dist[u] < 0]
            dist[level] = h + 1
    return out


def _graph(name):
    if name == "bipartite":  # every row of 600 entries, joined completely: any item brings the bits
        return _csr(1200, np.repeat(np.arange(600), 600), np.tile(600 + np.arange(600), 600))
    if name == "hubs":       # rows of 256, 257, 512, 513 and 3000 entries, chained by their last leaves
        a, b, at = [], [], 5
        for h, deg in enumerate([256, 257, 512, 513, 3000]):
            a += [h] * deg
            b += range(at, at + deg)
            at += deg - 1    # the next hub shares this one's last leaf
        return _csr(at + 1, np.array(a), np.array(b))
    n = 700                  # "complete": every row one entry short of three items
    i, j = np.triu_indices(n, 1)
    return _csr(n, i, j)


@pytest.mark.parametrize("name", ["bipartite", "hubs", "complete"])
@pytest.mark.parametrize("n_src", [1, 40, 300, 1025])
def test_sizes_on_rows_of_several_items(name, n_src):
    rowp, cols = _graph(name)
    n = len(rowp) - 1
    rng = np.random.default_rng(n_src)
    src = rng.integers(0, n, n_src).astype(np.int32)
    pred = (rng.random(n) < 0.7).astype(np.uint8)
    g = fl.Graph(rowp, cols)
    got = g.ball_sizes(src, 5, pred)
    some = np.unique(np.linspace(0, n_src - 1, 12).astype(int))
    assert np.array_equal(got[some], _sizes(rowp, cols, src[some], 5, pred))
    assert np.array_equal(got, np.stack([got[np.flatnonzero(src == s)[0]] for s in src]))  # equal sources, equal rows
    g.close()
