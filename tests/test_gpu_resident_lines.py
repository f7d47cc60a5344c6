"""Which graphs run their MIS and BFS as resident kernels: sparse graphs, whose
rows are work items of a few entries, on both sides of the lines on items and on
the ball radius, with the results of the host-driven rounds; batches on both
sides of theirs, with the results of plain solves."""
import numpy as np
import pytest

import flsynth
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _phases(g, cost, client):
    s = fl.Solve(g)
    s.compute_radii(cost, client)
    g.profile_reset()
    op, _ = s.open_facilities()
    mis = g.profile_query("mis")["launches"]
    g.profile_reset()
    a, d = s.assign_clients()
    bfs = g.profile_query("bfs")["launches"]
    log = s.mis_log()
    s.close()
    return (op, a, d), mis == 1, bfs == 1, int(log[log[:, 1] == 3][:, 2].max())


def _grid(w, h):
    v = np.arange(w * h).reshape(h, w)
    a = np.concatenate([v[:, :-1].ravel(), v[:-1].ravel()])
    b = np.concatenate([v[:, 1:].ravel(), v[1:].ravel()])
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    rowp = np.zeros(w * h + 1, np.int64)
    rowp[1:] = np.cumsum(np.bincount(src, minlength=w * h))
    return rowp, dst[np.argsort(src, kind="stable")].astype(np.int32)


def _check(g, cost, client, mis, bfs):
    g.profile(True)
    g.set_schedule(dense_div=8)
    got, mis_one, bfs_one, top = _phases(g, cost, client)
    assert (mis_one, bfs_one) == (mis, bfs), top
    g.set_schedule(dense_div=9)  # host-driven
    want, mis_one, bfs_one, _ = _phases(g, cost, client)
    assert not mis_one and not bfs_one
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
    return top


# items = vertices, below and above the line
@pytest.mark.parametrize("n,resident", [(1_550_000, True), (1_600_000, False)])
def test_line_on_items(n, resident):
    rowp, cols = flsynth.er(n, n, 8)
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    for cost in (20.0, 1.0e4):
        assert _check(g, np.full(n, cost), flsynth.bernoulli(n, 2, 0.7), resident, resident) <= 64
    g.close()


# balls of more than 64 hops, below and above their line
@pytest.mark.parametrize("side,mis", [(901, True), (1101, False)])
def test_line_of_large_balls(side, mis):
    rowp, cols = _grid(side, side + 8)
    n = len(rowp) - 1
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    assert _check(g, np.full(n, 3.0e4), np.ones(n, np.uint8), mis, True) > 64
    assert _check(g, np.full(n, 20.0), np.ones(n, np.uint8), True, True) <= 64
    g.close()


@pytest.mark.parametrize("n", [1_550_000, 1_600_000])
def test_batches_on_both_sides(n):
    per = n // 10
    rowp, cols = flsynth.er(per, per, 8)
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    b = fl.Batch.replicas(g, 10)
    cost = np.concatenate([np.full(per, 10.0 * (i + 1)) for i in range(10)])
    client = np.concatenate([flsynth.bernoulli(per, i, 0.3) for i in range(10)])
    got = b.solve(4, 3, cost, client)
    s = fl.Solve(g)
    for i in (0, 9):
        s.compute_radii(cost[i * per:(i + 1) * per], client[i * per:(i + 1) * per])
        op, _ = s.open_facilities()
        a, d = s.assign_clients()
        for key, want in (("open", op), ("assign", a), ("dist", d)):
            assert np.array_equal(got[key][i * per:(i + 1) * per], want), (i, key)
    s.close()
    b.close()
    g.close()
