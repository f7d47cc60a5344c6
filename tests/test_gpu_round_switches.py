"""Push and pull rounds driven by the host on graphs that would run their MIS and
BFS as resident kernels: a schedule that sets dense_div or edge_div gets the
rounds that these switch, on hubs cut into segments and on graphs made of parts
(uneven ones, parts of very different ball radii, more parts than a block's
table of radii holds), with the results of the resident kernels and the oracle."""
import numpy as np
import pytest

import brute
import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu

PUSH = dict(dense_div=1, edge_div=1)        # push unless the frontier is everything
PULL = dict(dense_div=1024, edge_div=1024)  # pull almost always
MIXED = dict(dense_div=8, edge_div=15)
FULL = dict(hop_group=0, sparse_div=16, graph_bfs=0, level_cap=0)


def _two_hubs():
    edges = [(0, i) for i in range(1, 6001)] + [(6001, i) for i in range(3500, 6500)]
    edges += [(i, i + 1) for i in range(6500, 8990)]
    rowp, cols = brute.csr_from_edges(9000, edges)
    fac = flsynth.bernoulli(9000, 22, 0.2)
    fac[[0, 6001, 8500]] = 1
    return rowp, cols, flsynth.loguniform(9000, 23, 3.0, 3000.0, fac), flsynth.bernoulli(9000, 21, 0.7)


def _rmat():
    rowp, cols = flsynth.rmat(13, 16, 88)
    n = len(rowp) - 1
    return rowp, cols, flsynth.loguniform(n, 5, 5.0, 500.0), flsynth.bernoulli(n, 6, 0.6)


@pytest.mark.parametrize("name", ["hubs", "rmat"])
def test_switches_take_effect_on_small_graphs(name):
    rowp, cols, cost, client = _two_hubs() if name == "hubs" else _rmat()
    want = oracle.solve(rowp, cols, 16, 5, cost, client)
    g = fl.Graph(rowp, cols)
    for sched in (PUSH, MIXED, PULL):
        g.set_schedule(**sched)
        g.build_sketches(16, 5)
        s = fl.Solve(g)
        s.compute_radii(cost, client)
        op, no = s.open_facilities()
        a, d = s.assign_clients()
        log = s.mis_log()
        rounds = set(log[np.isin(log[:, 1], (0, 1))][:, 4].tolist())
        assert sched is MIXED or (1 if sched is PULL else 0) in rounds, sched
        assert no == want["n_open"]
        for key, got in (("open", op), ("assign", a), ("dist", d)):
            assert np.array_equal(got, want[key]), (sched, key)
        s.close()
    g.close()


def _uneven():
    """(rowp, cols, cost, client) per part: ball radii from 0 to above 255."""
    parts = []
    for j, (n, deg) in enumerate([(3000, 9.0), (20000, 6.0), (400, 14.0)]):
        w = flsynth.small_er(n, deg, 300 + j)
        parts.append((w.rowp, w.cols, flsynth.loguniform(n, 40 + j, 2.0, 400.0, flsynth.bernoulli(n, 50 + j, 0.6)),
                      flsynth.bernoulli(n, 60 + j, 0.7)))
    rowp, cols = brute.csr_from_edges(700, [(i, i + 1) for i in range(699)])
    cost = np.full(700, np.inf)
    cost[[0, 350, 699]] = 1.0e5
    parts.append((rowp, cols, cost, np.ones(700, np.uint8)))
    rowp, cols = flsynth.er(500, 1000, 6)
    parts.append((rowp, cols, np.full(500, 0.25), np.ones(500, np.uint8)))
    parts.append((*_rmat()[:2], np.full(8192, 60.0), flsynth.bernoulli(8192, 9, 0.1)))
    parts.append((np.zeros(6, np.int64), np.zeros(0, np.int32), np.full(5, 3.0), np.ones(5, np.uint8)))
    return parts


def _many():
    """1100 small parts, constant costs (equal radii across parts)."""
    parts = []
    for i in range(1100):
        n = 20 + i % 23
        rowp, cols = flsynth.er(n, 2 * n, i % 37)
        parts.append((rowp, cols, np.full(n, [0.5, 4.0, 40.0][i % 3]), np.ones(n, np.uint8)))
    return parts


@pytest.mark.parametrize("make", [_uneven, _many])
@pytest.mark.parametrize("k", [4, 32])
def test_union_rounds(make, k):
    parts = make()
    cost, client = np.concatenate([p[2] for p in parts]), np.concatenate([p[3] for p in parts])
    b = fl.Batch.union([p[:2] for p in parts])
    base = b.solve(k, 3, cost, client)
    for sched in (PUSH, MIXED, PULL):
        b.set_schedule(dict(FULL, **sched))
        got = b.solve(k, 3, cost, client)
        for key in ("open", "assign", "dist", "n_open", "dist_sum", "n_unserved"):
            assert np.array_equal(got[key], base[key]), (sched, key)
    b.close()
    lo = 0
    for i, (rowp, cols, c, m) in enumerate(parts):
        hi = lo + len(c)
        if i % 100 < 8:
            want = oracle.solve(rowp, cols, k, 3, c, m)
            for key in ("open", "assign", "dist"):
                assert np.array_equal(base[key][lo:hi], want[key]), (i, key)
        lo = hi


@pytest.mark.parametrize("inst,sched", [(3, PUSH), (3, MIXED), (3, PULL), (30, {})])  # 30: above the resident size
def test_replica_rounds(inst, sched):
    rowp, cols = flsynth.rmat(14, 16, 515)
    n = len(rowp) - 1
    g = fl.Graph(rowp, cols)
    g.build_sketches(16, 5)
    costs = [np.where(flsynth.bernoulli(n, 1000 + i, 0.3) > 0, 5.0 * (i % 5 + 1) ** 2, np.inf) for i in range(inst)]
    clients = [flsynth.bernoulli(n, 1020 + i, 0.05 + 0.1 * (i % 6)) for i in range(inst)]
    b = fl.Batch.replicas(g, inst)
    if sched:
        b.set_schedule(dict(FULL, **sched))
    assert inst < 30 or inst * len(cols) > 10 * 2 ** 20
    for active in (inst, 2):
        got = b.solve(16, 5, np.concatenate(costs[:active]), np.concatenate(clients[:active]), n_active=active)
        for i in sorted({0, 1, active // 2, active - 1}):
            want = fl.solve(rowp, cols, 16, 5, costs[i], clients[i])
            for key in ("open", "assign", "dist"):
                assert np.array_equal(got[key][i * n:(i + 1) * n], want[key]), (active, i, key)
    b.close()
    g.close()
