"""MoCHy-A+ without the line graph, bitmaps in order of size (needs a GB300):
raw counts must equal MoCHy-A+ on the line graph bit for bit where the scan's
cases change: counts of 4 to 7 and of 8 or more bitmap nodes, list nodes
only, every size class for small and large theta, scans cut into parts, and
the budget just below and just above what both sets of bitmaps take.
"""
import numpy as np
import pytest

import oracle
from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu

# many hubs in long hyperedges; sizes 2 to 60; hyperedges of list nodes only;
# more hyperedges than one part of a scan
DEEP = synth.HypergraphSpec(160, 1200, 2, 60, "powerlaw", 1.2, "zipf", 1.0, seed=11)
FLAT = synth.HypergraphSpec(4000, 3000, 2, 6, "uniform", 0.0, "uniform", 0.0, seed=12)
LONG = synth.HypergraphSpec(20000, 70001, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=13)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("spec,theta", [(DEEP, 1), (DEEP, 2), (DEEP, 9), (DEEP, 60), (FLAT, 1)])
def test_counts_equal_the_oracle(spec, theta):
    off, nodes = synth.generate(spec)
    with B.Context(theta=theta) as c:
        c.load(spec.n_nodes, off, nodes)
        got = c.count_sampled_onthefly(1500, 6)
    ref = oracle.count_sampled(off, nodes, oracle.A_PLUS, 1500, 6, theta=theta)
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("samples", [1, 33, 5000])
def test_cut_scans_equal_the_line_graph(samples):
    off, nodes = synth.generate(LONG)
    with B.Context() as c:
        c.load(LONG.n_nodes, off, nodes)
        got = c.count_sampled_onthefly(samples, 19)
        c.project()
        ref = c.count_sampled(B.MOCHY_A_PLUS, samples, 19)
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)


def test_more_draws_than_a_launch_takes():
    off, nodes = synth.generate(FLAT)
    with B.Context() as c:
        c.load(FLAT.n_nodes, off, nodes)
        got = c.count_sampled_onthefly(70_001, 23)
        c.project()
        ref = c.count_sampled(B.MOCHY_A_PLUS, 70_001, 23)
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("both", [0, 1])
def test_budget_of_one_or_both_bitmaps(both):
    off, nodes = synth.generate(DEEP)
    words = ((len(off) - 1 + 31) // 32 + 3) // 4 * 4
    hubs = int((np.bincount(nodes) >= 16).sum())
    need = hubs * (2 * words + 4 * 65) * 4
    with B.Context() as c:
        c.load(DEEP.n_nodes, off, nodes)
        got = c.count_sampled_onthefly(700, 8, need - 1 + both)
    ref = oracle.count_sampled(off, nodes, oracle.A_PLUS, 700, 8)
    for a, b in zip(got[:4], ref):
        assert np.array_equal(a, b)
