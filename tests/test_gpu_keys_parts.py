"""Key order in unions of parts: a local id has one priority in every part, so
equal radii give runs of equal keys as long as the number of parts."""
import time

import numpy as np
import pytest

import brute
import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


# two local ids of equal radii, joined by an edge, whose priorities agree in the top half
@pytest.mark.parametrize("seed,a,b", [(646, 244, 817), (4835, 780, 937)])
@pytest.mark.parametrize("parts", [17, 32, 33, 70, 1100])  # runs of 2 x parts around the limit of 64
def test_two_ids_that_agree_in_the_top_half(seed, a, b, parts):
    assert oracle.priority(seed, a) >> 32 == oracle.priority(seed, b) >> 32
    rowp, cols = brute.csr_from_edges(1000, [(a, b)])
    cost, client = np.full(1000, 3.0), np.ones(1000, np.uint8)
    want = oracle.solve(rowp, cols, 4, seed, cost, client)
    assert want["open"][a] + want["open"][b] == 1
    u = fl.Batch.union([(rowp, cols)] * parts)
    got = u.solve(4, seed, np.tile(cost, parts), np.tile(client, parts))
    for key in ("open", "assign", "dist"):
        assert (got[key].reshape(parts, 1000) == want[key]).all(), key
    u.close()


def _pass_ms(graphs, n):
    import torch
    parts = len(graphs)
    u = fl.Batch.union(graphs)
    cost = torch.full((parts * n,), 20.0, dtype=torch.float64, device="cuda")
    client = torch.ones(parts * n, dtype=torch.uint8, device="cuda")
    ms = []
    for _ in range(6):
        torch.cuda.synchronize()
        t = time.perf_counter()
        u.solve(8, 3, cost, client)
        torch.cuda.synchronize()
        ms.append((time.perf_counter() - t) * 1e3)
    u.close()
    return min(ms)


def test_equal_parts_take_no_longer_than_different_ones():
    # ordered by one thread per run, 60,000 equal parts took four times as long as the others
    n, parts = 40, 60_000
    distinct = [flsynth.er(n, 2 * n, i) for i in range(64)]
    mixed = _pass_ms([distinct[i % 64] for i in range(parts)], n)
    equal = _pass_ms([distinct[0]] * parts, n)
    assert equal < 2.0 * mixed, (equal, mixed)
