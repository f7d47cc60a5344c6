"""Key order of the candidates on the GPU (radius, then priority) at the sizes
where its method changes: counting up to 16384 candidates, the radix sort above,
with distinct radii and with long runs of equal ones, against the oracle."""
import numpy as np
import pytest

import flsynth
import oracle
import paper_1503_03635_gb300 as fl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cost", ["equal", "few", "distinct"])
@pytest.mark.parametrize("m", [1, 2, 63, 513, 16384, 16385, 3 * 3072 * 2, 25_001])
def test_open_set_matches_the_oracle(m, cost):
    n = 26_000
    rowp, cols = flsynth.er(n, 2 * n, 900 + m)
    fac = np.zeros(n, np.uint8)
    fac[np.argsort(flsynth.hashes(n, m))[:m]] = 1
    val = {"equal": np.full(n, 7.5), "few": 5.0 + flsynth.hashes(n, 3).astype(np.float64) % 3,
           "distinct": flsynth.loguniform(n, 4, 5.0, 500.0)}[cost]
    c = np.where(fac > 0, val, np.inf)
    client = np.ones(n, np.uint8)  # every facility reaches a client (itself): m candidates
    got = fl.solve(rowp, cols, 4, 3, c, client)
    want = oracle.solve(rowp, cols, 4, 3, c, client)
    assert got["mis"]["candidates"] == m
    assert np.array_equal(got["open"], want["open"])
    assert np.array_equal(got["assign"], want["assign"])
    got["solve"].close()
    got["graph"].close()
