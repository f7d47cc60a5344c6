"""A time step of a weighted sweep sends no arrival past a label that the same step
is about to lower: every such arrival is one more time to run."""
import numpy as np
import pytest

import brute
import flsynth
import paper_1503_03635_gb300 as fl
from test_gpu_weighted import _compare


@pytest.mark.gpu
def test_sources_of_time_zero_send_nothing_to_each_other():
    # every vertex of a star is open, and the leaves' lengths are all different: only time 0 has arrivals that
    # count, but a leaf that pushes before the hub is drained sends it one at a time of its own, and so does the hub
    n = 1000
    edges = [(0, i) for i in range(1, n)]
    rowp, cols = brute.csr_from_edges(n, edges)
    src = np.repeat(np.arange(n), np.diff(rowp))
    lengths = (5 * np.maximum(src, cols) + 1).astype(np.int32)
    g = fl.Graph(rowp, cols, lengths=lengths)
    g.build_sketches(8, 3)
    s = fl.Solve(g)
    s.compute_radii(np.full(n, 0.5), np.ones(n, np.uint8))  # balls of radius 0: every facility opens
    _, n_open = s.open_facilities()
    assert n_open == n
    g.profile(True)
    ms = []
    for _ in range(6):
        g.profile_reset()
        a, d = s.assign_clients()
        ms.append(g.profile_query("bfs")["ms"])
        assert np.array_equal(a, np.arange(n)) and (d == 0).all()
    assert min(ms) < 0.5  # 1.3 to 2.7 ms with some hundred superfluous times
    s.close()
    g.close()


# many sources and one arrival time for most: constant costs (the cover's facilities enter together), unit and
# equal lengths, all open or nearly so
@pytest.mark.gpu
@pytest.mark.parametrize("length", [1, 7, 5000])
@pytest.mark.parametrize("cost", [0.5, 3.0, 4.0e4])
def test_mass_arrivals_match_the_oracle(length, cost):
    n = 700
    rowp, cols = flsynth.er(n, 2100, 4)
    lengths = np.full(len(cols), length, np.int32)
    _compare(rowp, cols, lengths, 8, 3, np.full(n, cost), flsynth.bernoulli(n, 5, 0.8))
