"""Exact ball sizes and radii where the sweeps can go wrong: rows at the limits
between the kernels and work items (32, 256 and 512 entries), numbers of sources
around the sweep widths, one source listed many times."""
import numpy as np
import pytest

import brute
import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _bfs_sizes(rowp, cols, src, D, pred):
    out = np.zeros((len(src), D + 1), np.int64)
    for i, s in enumerate(src):
        dist = np.full(len(rowp) - 1, -1)
        dist[s], level = 0, [s]
        for d in range(1, D + 1):
            nxt = []
            for v in level:
                for u in cols[rowp[v]:rowp[v + 1]]:
                    if dist[u] < 0:
                        dist[u] = d
                        nxt.append(u)
            level = nxt
        for d in range(D + 1):
            out[i, d] = np.sum((dist >= 0) & (dist <= d) & (pred > 0))
    return out


@pytest.mark.parametrize("deg", [32, 33, 256, 257, 512, 513, 1025, 2100])
def test_row_limits(deg):
    n = 2 * deg + 2
    rowp, cols = brute.csr_from_edges(n, [(0, 2 + i) for i in range(deg)] + [(1, 2 + deg // 2 + i) for i in range(deg)])
    src = np.array([0, 1, 2, n - 1, 2 + deg // 2, 0], np.int32)
    pred = flsynth.bernoulli(n, 5, 0.5)
    g = fl.Graph(rowp, cols)
    assert np.array_equal(g.ball_sizes(src, 5, pred), _bfs_sizes(rowp, cols, src, 5, pred))
    g.close()


@pytest.mark.parametrize("n_src", [1, 64, 256, 257, 512, 513, 1024, 1025, 1400])
def test_sweep_widths(n_src):
    rowp, cols = flsynth.rmat(10, 8, 33)
    n = len(rowp) - 1
    base = np.arange(n, dtype=np.int32)[flsynth.hashes(n, 3).argsort()][:40]
    src = base[np.arange(n_src) % 40]
    pred = flsynth.bernoulli(n, 6, 0.4)
    g = fl.Graph(rowp, cols)
    want = _bfs_sizes(rowp, cols, base, 6, pred)
    assert np.array_equal(g.ball_sizes(src, 6, pred), want[np.arange(n_src) % 40])
    g.close()


@pytest.mark.parametrize("facs", [200, 600, 1300])
def test_exact_radii_of_many_facilities(facs):
    rowp, cols = flsynth.rmat(11, 8, 34)
    n = len(rowp) - 1
    cost = np.full(n, np.inf)
    cost[flsynth.hashes(n, 8).argsort()[:facs]] = flsynth.loguniform(n, 9, 5.0, 400.0)[:facs]
    client = flsynth.bernoulli(n, 10, 0.5)
    og = oracle.Graph(rowp, cols)
    want = og.exact_radii(cost, client)
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 1)
    s = fl.Solve(g)
    got = s.compute_radii_exact(cost, client)
    fin = np.isfinite(want)
    assert np.array_equal(np.isfinite(got), fin) and np.array_equal(got[fin], want[fin])
    s.close()
    g.close()
    og.close()
