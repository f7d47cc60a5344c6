"""Which graphs run their MIS and BFS as resident kernels: sparse graphs, whose
rows are work items of a few entries, on both sides of the lines on items and on
the ball radius, with the results of the host-driven rounds."""
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


# items = vertices: below the BFS line, between it and the MIS line, above both
@pytest.mark.parametrize("n,small,wide,bfs", [(700_000, True, True, True), (1_200_000, True, False, False),
                                              (1_700_000, False, False, False)])
def test_lines_on_items(n, small, wide, bfs):
    rowp, cols = flsynth.er(n, n, 8)
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 3)
    g.profile(True)
    for cost, resident in ((20.0, small), (1.0e4, wide)):
        c, m = np.full(n, cost), flsynth.bernoulli(n, 2, 0.7)
        g.set_schedule(dense_div=8)
        got, mis_one, bfs_one, top = _phases(g, c, m)
        assert (top > 16) == (cost > 20.0)
        assert (mis_one, bfs_one) == (resident, bfs), (cost, top)
        g.set_schedule(dense_div=9)  # host-driven
        want, mis_one, bfs_one, _ = _phases(g, c, m)
        assert not mis_one and not bfs_one
        for x, y in zip(got, want):
            assert np.array_equal(x, y), cost
    g.close()
