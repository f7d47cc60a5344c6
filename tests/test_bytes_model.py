"""The bytes models of the sketch merge charge what the kernels hold: ordinals of
4 bytes in sketches and delta lists."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_model_of_the_bench():
    from bench import merge_model_bytes

    # a path of three vertices, k = 2, hop 1: 4 edge-merges of one ordinal each into 3 vertices, 4 entries gained
    hop = dict(edge_merges=4, merging=3, delta_sum=4, delta_read=0, new_entries=4)
    rows, columns, deltas, sketches, entries = 3 * 8, 4 * 4, 4 * 4, 3 * 2 * (4 + 4), 4 * 12
    assert merge_model_bytes([hop], 2) == rows + columns + deltas + sketches + entries
    assert merge_model_bytes([hop, hop], 2) == 2 * merge_model_bytes([hop], 2)


@pytest.mark.gpu
@pytest.mark.parametrize("k", [4, 32])
def test_bytes_of_the_merge_class(k):
    import flsynth
    import paper_1503_03635_gb300 as fl

    rowp, cols = flsynth.rmat(13, 16, 9)
    g = fl.Graph(rowp, cols)
    g.profile(True)
    g.profile_reset()
    g.build_sketches(k, 3)
    got = g.profile_query("sketch_merge")["alg_bytes"]
    want = sum(8 * h["merging"] + 4 * h["edge_merges"] + 8 * h["delta_read"] + 8 * k * h["merging"]
               + 12 * h["new_entries"] for h in g.hop_model())
    assert np.isclose(got, want, rtol=1e-12)
    g.close()
