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


def _zipf(edges, seed):
    spec = synth.HypergraphSpec(max(edges // 2, 64), edges, 2, 25, "powerlaw", 2.5, "zipf", 1.0,
                                seed=seed)
    return (spec.n_nodes, *synth.generate(spec))


def _one_set_of_bitmaps(g, budget):
    """Bytes of one set of bitmaps within a quarter of the budget, size planes,
    prefix and two words a hyperedge, each rounded to 256."""
    n, off, nodes = g
    E = len(off) - 1
    words = max((E + 31) // 32, 1)
    pop = int((np.bincount(nodes, minlength=n) >= max(words // 32, 16)).sum())
    maps = max(min(pop, budget // 4 // (4 * words)), 1)
    return sum((b + 255) & ~255 for b in (4 * n, 4 * maps, 4 * words * maps, 16 * words,
                                          8 * (E + 1), 8 * E, 8 * E))


@pytest.mark.parametrize("g", [_zipf(4001, 5), _uniform(300, 90, 6), _uniform(60, 21, 7)],
                         ids=["zipf4001", "uniform90", "uniform21"])
def test_least_budget_is_that_of_one_set_of_bitmaps(g):
    """Neither the second set of bitmaps nor the draws of a launch make a call
    fail whose budget holds one set."""
    with B.Context() as c:
        c.load(*g)
        loaded = B.mochy_device_bytes(c.h)
        ref = c.count_sampled_onthefly(500, 8)
    budget = loaded
    while loaded + _one_set_of_bitmaps(g, budget) > budget:
        budget += 256
    with B.Context(budget=budget) as c:
        c.load(*g)
        got = c.count_sampled_onthefly(500, 8)
        assert B.mochy_device_bytes(c.h) <= budget
    assert got[4] == ref[4]
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)
