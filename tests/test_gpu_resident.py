"""The resident MIS and BFS kernels of small graphs against the oracle where
they can go wrong: rows at the edges of their work items (64 entries), more
greedy rounds than one launch runs, ball radii above the kernel's limit, balls
of radius 0, and the size above which graphs take the host-driven rounds."""
import numpy as np
import pytest

import brute
import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _check(rowp, cols, k, cost, client):
    got = fl.solve(rowp, cols, k, 5, cost, client)
    want = oracle.solve(rowp, cols, k, 5, cost, client)
    for key in ("open", "assign", "dist"):
        assert np.array_equal(got[key], want[key]), key
    rounds = got["mis"]["mis_rounds"]
    log = got["solve"].mis_log()
    tot = log[log[:, 1] == 3]
    assert len(tot) == rounds and tot[:, 4].sum() == got["mis"]["candidates"]
    got["solve"].close()
    got["graph"].close()
    return rounds


@pytest.mark.parametrize("deg", [1, 63, 64, 65, 128, 129, 2048, 2049])
def test_rows_at_item_edges(deg):
    # two hubs of `deg` entries sharing half of their leaves
    n = 2 * deg + 2
    edges = [(0, 2 + i) for i in range(deg)] + [(1, 2 + deg // 2 + i) for i in range(deg)]
    rowp, cols = brute.csr_from_edges(n, edges)
    _check(rowp, cols, 8, flsynth.loguniform(n, deg, 1.5, 300.0), flsynth.bernoulli(n, 9, 0.7))


@pytest.mark.parametrize("n", [40, 900])
def test_more_greedy_rounds_than_one_launch(n):
    rowp, cols = brute.csr_from_edges(n, [(i, i + 1) for i in range(n - 1)])
    rounds = _check(rowp, cols, 32, 2.5 + 0.003 * np.arange(n), np.ones(n, np.uint8))
    assert n < 900 or rounds > 32


@pytest.mark.parametrize("cost", [1.0e5, 6.0e5, 5.0e6])
def test_ball_radii_around_the_kernel_limit(cost):
    n = 2600
    rowp, cols = brute.csr_from_edges(n, [(i, i + 1) for i in range(n - 1)])
    c = np.full(n, np.inf)
    c[[0, 700, 1300, 2599]] = [cost, 2 * cost, cost, 0.5 * cost]
    _check(rowp, cols, 32, c, np.ones(n, np.uint8))


def test_balls_of_radius_zero():
    n = 500
    rowp, cols = flsynth.er(n, 1000, 6)
    _check(rowp, cols, 16, np.full(n, 0.25), np.ones(n, np.uint8))


@pytest.mark.parametrize("M", [5_242_000, 5_243_000])  # 2M entries: below and above 10 x 2^20
def test_both_sides_of_the_size_limit(M):
    n = 300_000
    rowp, cols = flsynth.er(n, M, 8)
    _check(rowp, cols, 4, np.full(n, 30.0), flsynth.bernoulli(n, 2, 0.3))
