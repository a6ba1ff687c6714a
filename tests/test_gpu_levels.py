"""The exact count by levels of overlap against the oracle, where its tables,
its split of rows and its hub and light nodes can go wrong: overlaps past the
bit fields of the level 3 table, hyperedges past 32 nodes (no node masks), rows
with just few and just many heavy pairs, graphs of hubs only and of light nodes
only, every threshold it covers and the first it does not."""
import numpy as np
import pytest

import oracle
from paper_2310_15668_gb300 import binding as B, synth
from . import _util

pytestmark = pytest.mark.gpu


def _random(n, e, lo, hi, seed):
    rng = np.random.default_rng(seed)
    sets = {tuple(sorted(rng.choice(n, rng.integers(lo, hi + 1), replace=False).tolist()))
            for _ in range(e)}
    return (n, *_util.csr_from_sets(sorted(sets)))


def _shared_pair(copies):
    """`copies` hyperedges that share the node pair {0, 1}, each with one node
    of its own (so each has copies - 1 heavy pairs), and some singletons,
    pairs and triples around them."""
    sets = [(0, 1, 2 + i) for i in range(copies)]
    sets += [(0,), (1, 2), (2, 3), (0, 2, 3), (1, 3, 4, 5)]
    return (copies + 2, *_util.csr_from_sets(sets))


def _clusters():
    spec = synth.HypergraphSpec(300, 400, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=4)
    off, nodes = synth.generate(spec)
    off, nodes = synth.plant_cluster(off, nodes, 120, 40, 24, 8, 22, seed=5)
    return (300, off, nodes)


def _spec(n, e, **kw):
    spec = synth.HypergraphSpec(n, e, **kw)
    return (n, *synth.generate(spec))


GRAPHS = {
    "all_hubs": lambda: _random(40, 500, 2, 6, 1),
    "all_light": lambda: _random(3000, 1500, 2, 5, 2),
    "few_48": lambda: _shared_pair(49),
    "many_49": lambda: _shared_pair(50),
    "stage_65": lambda: _shared_pair(66),
    "wide": lambda: _random(90, 140, 20, 63, 3),
    "size_32_33": lambda: _random(60, 120, 30, 35, 6),
    "clusters": _clusters,
    "zipf1k": lambda: _spec(500, 1000, seed=9),
    "singletons": lambda: _random(12, 60, 1, 3, 7),
}


@pytest.mark.parametrize("theta", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_levels_match_oracle(name, theta):
    n, off, nodes = GRAPHS[name]()
    with B.Context(theta=theta) as c:
        c.load(n, off, nodes)
        c.project()
        B.mochy_trace(c.h, 1)
        h, h3 = c.count_exact()
        phases = B.mochy_trace_read(c.h)["phases_ms"]
        again = c.count_exact()
    oh, o3 = oracle.count_exact(off, nodes, theta=theta)
    assert np.array_equal(h3, o3) and np.array_equal(h, oh)
    assert np.array_equal(again[0], h) and np.array_equal(again[1], h3)
    assert ("level 3" in phases) == (theta <= 4)


@pytest.mark.parametrize("k,thr", [(2, ()), (3, (1,)), (3, (4,)), (3, (5,)), (4, (1, 2)),
                                   (4, (2, 4)), (4, (1, 5))])
@pytest.mark.parametrize("name", ["all_hubs", "clusters", "size_32_33"])
def test_kh_motifs_by_levels_match_oracle(name, k, thr):
    """Thresholds up to 4 are counted by levels, larger ones by the scan; an
    exact count in between keeps its own tables."""
    n, off, nodes = GRAPHS[name]()
    with B.Context() as c:
        c.load(n, off, nodes)
        c.project()
        first = c.count_kh(k, thr)
        h, h3 = c.count_exact()
        second = c.count_kh(k, thr)
    o = oracle.count_exact_kh(off, nodes, k, thr)
    oh, o3 = oracle.count_exact(off, nodes)
    assert np.array_equal(h, oh) and np.array_equal(h3, o3)
    for got in (first, second):
        assert np.array_equal(got[0], o[0]) and np.array_equal(got[1], o[1])


def test_levels_in_a_batch_of_unlike_hypergraphs():
    """Units of a batch keep their own hubs, matrices and tables."""
    gs = [GRAPHS[k]() for k in ("all_hubs", "few_48", "clusters", "all_light", "zipf1k")]
    R = 2
    seeds = [3 + g for g in range(len(gs))]
    _, _, _, _, ch, c3, _, _ = B.mochy_profile_batch(gs, R, seeds)
    for g, (n, off, nodes) in enumerate(gs):
        o = oracle.profile(n, off, nodes, R, seeds[g])
        assert np.array_equal(ch[g], o["counts_h"]) and np.array_equal(c3[g], o["counts_3h"])


def test_levels_with_more_hubs_than_the_hub_matrix_holds():
    """About 5,400 nodes of degree 32 or more (the hub matrix holds 4,096):
    the others are counted as light nodes.  Against the per-hyperwedge scan."""
    n, off, nodes = _random(6000, 48000, 5, 5, 11)
    assert (np.bincount(nodes, minlength=n) >= 32).sum() > 4500
    got = []
    for kernel in (0, 1):
        with B.Context(exact_kernel=kernel) as c:
            c.load(n, off, nodes)
            c.project()
            got.append(c.count_exact())
    assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][0], got[1][0])
