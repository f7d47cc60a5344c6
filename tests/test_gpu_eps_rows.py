"""The resident event loop of the phase with eps > 0 against the oracle where it
can go wrong: rows at the length that a whole block takes (one or two in a
block's queue; more than it holds: test_gpu_eps_queue.py), components without
facilities or clients, and the level cap."""
import numpy as np
import pytest

import brute
import flsynth
import paper_1503_03635_gb300 as fl
from test_gpu_eps import _compare

pytestmark = pytest.mark.gpu


def _hubs(n_hubs, deg):
    """Hubs whose leaves overlap by half."""
    edges = [(h, n_hubs + h * (deg // 2) + i) for h in range(n_hubs) for i in range(deg)]
    return brute.csr_from_edges(n_hubs + n_hubs * (deg // 2) + deg, edges)


@pytest.mark.parametrize("n_hubs,deg", [(2, 511), (2, 512), (2, 513), (160, 520), (1, 3000)])
@pytest.mark.parametrize("eps", [0.1, 1.0])
def test_rows_at_the_edges(n_hubs, deg, eps):
    rowp, cols = _hubs(n_hubs, deg)
    n = len(rowp) - 1
    fac = flsynth.bernoulli(n, 7, 0.05)
    fac[:n_hubs] = 1  # the hubs open too
    _compare(rowp, cols, 8, 3, eps, flsynth.loguniform(n, 8, 1.0, 40.0, fac), flsynth.bernoulli(n, 9, 0.6))


def test_components_without_facilities_or_clients():
    rowp, cols = brute.csr_from_edges(90, [(i, i + 1) for i in range(89) if i % 30 != 29])
    cost, client = np.full(90, np.inf), np.ones(90, np.uint8)
    cost[:60:7] = 3.0
    client[:30] = 0
    _compare(rowp, cols, 4, 2, 0.3, cost, client)


def test_level_cap_is_refused():
    rowp, cols = brute.csr_from_edges(40, [(i, i + 1) for i in range(39)])
    cost = np.full(40, np.inf)
    cost[0] = 1.0
    g = fl.Graph(rowp, cols)
    g.build_sketches(4, 1)
    s = fl.Solve(g)
    g.set_schedule(level_cap=20)
    with pytest.raises(fl.FLError) as e:
        s.open_facilities_eps(0.5, cost, np.ones(40, np.uint8))
    assert e.value.status == fl.FL_ETIMEOUT
    g.set_schedule(level_cap=40)
    s.open_facilities_eps(0.5, cost, np.ones(40, np.uint8))
    s.close()
    g.close()


@pytest.mark.parametrize("deg", [255, 256, 257, 769])
def test_gamma_over_rows_at_segment_edges(deg):
    # one facility, the leaf that comes last in the hubs' rows
    rowp, cols = _hubs(3, deg)
    n = len(rowp) - 1
    cost = np.full(n, np.inf)
    cost[n - 1] = 2.5
    _compare(rowp, cols, 8, 3, 0.2, cost, np.ones(n, np.uint8))
