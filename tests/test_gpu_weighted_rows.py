"""The weighted build and sweeps against the oracle where they can go
wrong: rows at the edges of the mark words and of the lengths that a whole
block and the whole grid take, more long rows than a block queues, more hubs
than blocks, one vertex, lengths that make the ring as short and as long as it
gets."""
import numpy as np
import pytest

import brute
import flsynth
import paper_1503_03635_gb300 as fl
from test_gpu_weighted import _compare

pytestmark = pytest.mark.gpu


def _hubs(n_hubs, deg):
    """Hubs whose leaves overlap by half."""
    edges = [(h, n_hubs + h * (deg // 2) + i) for h in range(n_hubs) for i in range(deg)]
    return brute.csr_from_edges(n_hubs + n_hubs * (deg // 2) + deg, edges)


@pytest.mark.parametrize("n_hubs,deg,hi", [(2, 31, 100), (3, 32, 7), (2, 33, 1), (2, 511, 100), (2, 512, 100),
                                           (2, 513, 3), (60, 600, 20), (1, 3000, 100)])
def test_rows_at_the_edges(n_hubs, deg, hi):
    rowp, cols = _hubs(n_hubs, deg)
    n = len(rowp) - 1
    w = flsynth.edge_weights(rowp, cols, 31, 1, hi)
    fac = flsynth.bernoulli(n, 7, 0.3)
    cost = flsynth.loguniform(n, 8, 5.0 * hi, 60.0 * hi, fac)
    _compare(rowp, cols, w, 8, 3, cost, flsynth.bernoulli(n, 9, 0.6))


@pytest.mark.parametrize("k", [2, 32])
def test_long_lengths_and_single_vertices(k):
    rowp, cols = brute.csr_from_edges(40, [(i, i + 1) for i in range(6)] + [(20, 21), (21, 22), (20, 22)])
    w = flsynth.edge_weights(rowp, cols, 5, 3000, 9000)
    cost = np.full(40, 20000.0)
    _compare(rowp, cols, w, k, 1, cost, np.ones(40, np.uint8))


@pytest.mark.parametrize("n_hubs,deg", [(2, 1023), (2, 1024), (2, 1025), (3, 4100)])
def test_hubs_posted_by_the_grid(n_hubs, deg):
    rowp, cols = _hubs(n_hubs, deg)
    w = flsynth.edge_weights(rowp, cols, 37, 1, 20)
    n = len(rowp) - 1
    _compare(rowp, cols, w, 12, 3, np.full(n, 80.0), flsynth.bernoulli(n, 9, 0.6))


def test_more_hubs_than_blocks():
    n_hubs, leaves = 160, 1040
    rowp, cols = brute.csr_from_edges(n_hubs + leaves, [(h, n_hubs + i) for h in range(n_hubs) for i in range(leaves)])
    n = len(rowp) - 1
    w = flsynth.edge_weights(rowp, cols, 41, 1, 50)
    _compare(rowp, cols, w, 16, 3, flsynth.loguniform(n, 8, 50.0, 2000.0), flsynth.bernoulli(n, 9, 0.6))


def test_more_rows_than_a_block_queues():
    # unit lengths: the unweighted build of the same graph
    rowp, cols = flsynth.er(24000, 24000 * 24, 6)
    out = []
    for lengths in (None, np.ones(len(cols), np.int32)):
        g = fl.Graph(rowp, cols, lengths=lengths)
        g.build_sketches(4, 3)
        out.append(g.export_ads())
        g.close()
    for key in ("gofs", "eofs", "ghop", "gcnt", "gcounted", "eid", "gwt"):
        assert np.array_equal(out[0][key], out[1][key]), key
