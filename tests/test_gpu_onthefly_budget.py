"""MoCHy-A+ without the line graph at the edges of its memory (needs a GB300):
hyperedge counts at which an array of one entry each ends on its block's last
byte, and budgets that hold one set of bitmaps, or none.
"""
import numpy as np
import pytest

from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _uniform(nodes, edges, seed):
    spec = synth.HypergraphSpec(nodes, edges, 2, 5, "uniform", 0.0, "uniform", 0.0, seed=seed)
    return (nodes, *synth.generate(spec))


@pytest.mark.parametrize("edges", [32 * 1024, 32 * 1025, 32 * 1025 + 1])
def test_scan_of_the_neighbours_at_multiples_of_32(edges):
    """8 (E + 1) bytes pass a multiple of 256 at E = 32 m."""
    n, off, nodes = _uniform(20000, edges, edges)
    assert len(off) - 1 == edges
    with B.Context() as c:
        c.load(n, off, nodes)
        got = c.count_sampled_onthefly(900, 4)
        nw, _ = c.project()
        ref = c.count_sampled(B.MOCHY_A_PLUS, 900, 4)
    assert got[4] == nw
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)
