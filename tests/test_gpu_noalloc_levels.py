"""The allocation-free assignment against a plain BFS where its levels can go
wrong: rows at the edges of the 32-row windows and of the 128-entry steps, thin frontiers
(push) and wide ones (pull), long rows in levels that pull, and graphs whose
entries do not fill one window.  (Long rows in levels that push:
test_gpu_noalloc_push.py.)"""
import numpy as np
import pytest

import brute
import flsynth
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


def _bfs(rowp, cols, is_open):
    n = len(rowp) - 1
    assign, dist = np.full(n, -1, np.int32), np.full(n, -1, np.int32)
    level = np.flatnonzero(is_open)
    assign[level], dist[level] = level, 0
    d = 0
    while len(level):
        d += 1
        best = {}
        for v in level:
            for u in cols[rowp[v]:rowp[v + 1]]:
                if dist[u] < 0:
                    best[u] = min(best.get(u, n), assign[v])
        for u, lab in best.items():
            assign[u], dist[u] = lab, d
        level = np.fromiter(best, np.int64, len(best))
    return assign, dist


def _hubs(n_hubs, deg, gap):
    """Hubs whose leaves overlap by half, with `gap` isolated vertices in front."""
    edges, first = [], gap + n_hubs
    for h in range(n_hubs):
        edges += [(gap + h, first + h * (deg // 2) + i) for i in range(deg)]
    return brute.csr_from_edges(first + n_hubs * (deg // 2) + deg, edges)


CASES = {
    "one": (np.zeros(2, np.int64), np.zeros(0, np.int32), [0]),
    "path": (*brute.csr_from_edges(2000, [(i, i + 1) for i in range(1999)]), [0, 1999, 700]),
    "row31": (*_hubs(3, 31, 31), [33]),
    "row32": (*_hubs(3, 32, 32), [36]),
    "row129": (*_hubs(4, 129, 1), [1, 3]),
    "row512": (*_hubs(2, 512, 0), [1]),
    "row513": (*_hubs(2, 513, 0), [0]),
    "queue": (*_hubs(600, 520, 5), list(range(5, 605, 2))),
    "rmat": (*flsynth.rmat(14, 16, 5), [3, 77, 9000]),
    "none": (*flsynth.rmat(10, 4, 5), []),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_levels_match_plain_bfs(name):
    import torch
    rowp, cols, opened = CASES[name]
    n = len(rowp) - 1
    is_open = np.zeros(n, np.uint8)
    is_open[opened] = 1
    want = _bfs(rowp, cols, is_open)
    to = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    a = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    d = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    for _ in range(2):
        fl.assign_nearest_noalloc(to(rowp), to(cols), to(is_open), a, d)
        assert np.array_equal(a.cpu().numpy(), want[0])
        assert np.array_equal(d.cpu().numpy(), want[1])
