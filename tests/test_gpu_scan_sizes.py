"""Prefix sums at the sizes where their launches change (needs a GB300): one
tile of 4,096 values, the first size of two tiles, the last size whose tiles
add up each other's sums and the first beyond.  The hypergraph is a path,
{i, i + 1} for each i: every prefix sum of loading and projecting it shows in
its line degrees, 2 but for the two ends.
"""
import numpy as np
import pytest

from paper_2310_15668_gb300 import binding as B

pytestmark = pytest.mark.gpu

TILE = 4096


@pytest.mark.parametrize("edges", [2, TILE - 1, TILE, TILE + 1, 3 * TILE + 5, TILE * 1024,
                                   TILE * 1024 + 1])
def test_path_line_graph(edges):
    off = 2 * np.arange(edges + 1, dtype=np.int64)
    nodes = (np.arange(edges, dtype=np.int32)[:, None] + np.arange(2, dtype=np.int32)).ravel()
    with B.Context() as c:
        c.load(edges + 1, off, nodes)
        n_wedges, max_degree = c.project()
        deg = c.line_degrees()
    ref = np.full(edges, 2, np.int64)
    ref[0] = ref[-1] = 1
    assert n_wedges == edges - 1 and max_degree == ref.max()
    assert np.array_equal(deg, ref)
