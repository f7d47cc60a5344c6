"""More long rows in one level of the eps phase's distance search than the blocks
queue (128 rows above 512 entries each): the rows left over are spread by a warp."""
import numpy as np
import pytest

import paper_1503_03635_gb300 as fl


@pytest.mark.gpu
def test_more_long_rows_than_the_blocks_queue():
    # 512 pads joined to every hub, a leaf per hub, pad 7 the only facility that opens: every hub is in the frontier
    # of level 2, 24,000 rows over at most 152 blocks, and each leaf is reached by its own hub alone; an isolated
    # facility without clients never opens (the phase ends with the last facility)
    pads, hubs, eps = 512, 24_000, 0.5
    assert hubs > 152 * 128
    n = pads + 2 * hubs + 1
    h = np.arange(pads, pads + hubs)
    src = np.concatenate([np.tile(np.arange(pads), hubs), h])
    dst = np.concatenate([np.repeat(h, pads), h + hubs])
    src, dst = np.concatenate([src, dst]), np.concatenate([dst, src])
    order = np.argsort(src, kind="stable")
    rowp = np.zeros(n + 1, np.int64)
    rowp[1:] = np.cumsum(np.bincount(src, minlength=n))
    cost = np.full(n, np.inf)
    cost[[7, n - 1]] = 2.0
    client = np.ones(n, np.uint8)
    client[n - 1] = 0
    got = fl.solve_eps(rowp, dst[order].astype(np.int32), 8, 3, eps, cost, client)
    dist = np.full(n, 2, np.int32)
    dist[7], dist[h], dist[n - 1] = 0, 1, -1
    assert np.array_equal(got["dist"], dist) and (got["assign"][:-1] == 7).all()
    # a client freezes at the first iteration, from the opening on, whose (1 + eps) alpha_j reaches its distance
    grid = [got["stats"]["alpha0"]]
    while grid[-1] < 10.0:
        grid.append(grid[-1] * (1.0 + eps))
    reach = (1.0 + eps) * np.array(grid)
    opened = int(got["fac_iter"][7])
    want = np.where(client > 0, np.maximum(opened, np.searchsorted(reach, dist.astype(np.float64))), -1)
    assert opened >= 1
    assert np.array_equal(got["cli_iter"], want)
    got["solve"].close()
    got["graph"].close()
