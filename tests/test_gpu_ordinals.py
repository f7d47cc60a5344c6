"""Sketches by ordinals against the oracle where the order of the ranks is made
in different ways or lists are merged at their limits: few vertices (counted),
many (sorted), every sketch width around the group widths, rows of one chunk
and a little more, and unions whose parts' sizes differ by much."""
import numpy as np
import pytest

import brute
import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _check(rowp, cols, k, seed, group=0):
    og = oracle.Graph(rowp, cols)
    og.build_sketches(k, seed)
    want, A = og.sketch(), og.ads(ranks=False)
    g = fl.Graph(rowp, cols)
    g.set_schedule(hop_group=group)
    g.build_sketches(k, seed)
    S, cnt = g.export_sketches()
    assert np.array_equal(cnt, want[1]) and np.array_equal(S, want[0])
    B = g.export_ads()
    for key in ("gofs", "eofs", "ghop", "gcnt", "gcounted", "eid"):
        assert np.array_equal(A[key], B[key]), key
    assert np.array_equal(A["gwt"].view(np.uint64), B["gwt"].view(np.uint64))
    g.close()
    og.close()


@pytest.mark.parametrize("n", [2, 63, 64, 65, 2048, 2049, 16384, 16385, 40000])
def test_counted_and_sorted_ranks(n):
    w = flsynth.small_er(n, 3.0, n)
    _check(w.rowp, w.cols, 8, 7)


@pytest.mark.parametrize("k", [2, 3, 15, 16, 17, 31, 32])
@pytest.mark.parametrize("group", [0, 32])
def test_sketch_widths(k, group):
    rowp, cols = flsynth.rmat(12, 12, 91)
    _check(rowp, cols, k, 2, group)


@pytest.mark.parametrize("deg", [15, 16, 17, 31, 32, 33, 64, 65])
def test_rows_at_chunk_edges(deg):
    n = 4 * deg + 9  # a circulant graph: every row holds 2 * deg entries, every list is full
    edges = [(i, (i + d) % n) for i in range(n) for d in range(1, deg + 1)]
    rowp, cols = brute.csr_from_edges(n, edges)
    _check(rowp, cols, 16, 4)
    _check(rowp, cols, 32, 4)


def test_union_of_uneven_parts():
    graphs = [(w.rowp, w.cols) for w in (flsynth.small_er(n, 5.0, n) for n in (3, 300, 20000, 70, 1500))]
    n = sum(len(r) - 1 for r, _ in graphs)
    cost, client = flsynth.loguniform(n, 5, 4.0, 90.0), flsynth.bernoulli(n, 6, 0.5)
    b = fl.Batch.union(graphs)
    res = b.solve(16, 9, cost, client)
    lo = 0
    for i, (rowp, cols) in enumerate(graphs):
        hi = lo + len(rowp) - 1
        want = oracle.solve(rowp, cols, 16, 9, cost[lo:hi], client[lo:hi])
        for key in ("open", "assign", "dist"):
            assert np.array_equal(res[key][lo:hi], want[key]), (i, key)
        lo = hi
    b.close()
