"""Replica batches of a relabelled graph whose vertex total is no multiple of 4:
the distances are staged behind one byte per vertex."""
import numpy as np
import pytest

import flsynth
import paper_1503_03635_gb300 as fl


def _odd_graph(n):
    """The first n vertices of an R-MAT graph with hubs."""
    rowp, cols = flsynth.rmat(12, 8, 21)
    src = np.repeat(np.arange(len(rowp) - 1), np.diff(rowp))
    keep = (src < n) & (cols < n)
    counts = np.bincount(src[keep], minlength=n)
    return np.concatenate([[0], np.cumsum(counts)]).astype(np.int64), cols[keep].astype(np.int32)


@pytest.mark.gpu
@pytest.mark.parametrize("n,inst", [(4001, 1), (4001, 2), (4001, 3), (4003, 4)])
def test_replicas_with_odd_totals(n, inst):
    rowp, cols = _odd_graph(n)
    g = fl.Graph(rowp, cols)
    g.build_sketches(8, 3)
    b = fl.Batch.replicas(g, inst)
    costs = [flsynth.loguniform(n, 40 + i, 5.0, 300.0) for i in range(inst)]
    clients = [flsynth.bernoulli(n, 60 + i, 0.5) for i in range(inst)]
    res = b.solve(8, 3, np.concatenate(costs), np.concatenate(clients))
    for i in range(inst):
        want = fl.solve(rowp, cols, 8, 3, costs[i], clients[i])
        for key in ("open", "assign", "dist"):
            assert np.array_equal(res[key][i * n:(i + 1) * n], want[key]), (key, i)
    b.close()
    g.close()
