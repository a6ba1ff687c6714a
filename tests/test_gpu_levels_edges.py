"""The exact count by levels of overlap at the limits of its structures (needs
a GB300), against the oracle.
"""
import time

import numpy as np
import pytest

import oracle
from paper_2310_15668_gb300 import binding as B, synth
from . import _util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _wide(n, e, lo, hi, seed):
    rng = np.random.default_rng(seed)
    sets = {tuple(sorted(rng.choice(n, rng.integers(lo, hi + 1), replace=False).tolist()))
            for _ in range(e)}
    return (n, *_util.csr_from_sets(sorted(sets)))


def _count(g, **kw):
    with B.Context(**kw) as c:
        c.load(*g)
        c.project()
        return c.count_exact()


def _distinct_tuples(g, theta, t_from):
    """Region sizes of the triples with t >= t_from common nodes and three
    overlaps of 2 or more, own regions capped at t + theta + 1, the members in
    any order: fewer than the level 3 tuples."""
    n, off, nodes = g
    E = len(off) - 1
    m = np.zeros((E, n), np.int32)
    for i in range(E):
        m[i, nodes[off[i]:off[i + 1]]] = 1
    om = m @ m.T
    size = m.sum(1)
    keys = set()
    for a in range(E):
        t = (m * m[a]) @ m.T
        b, k = np.triu_indices(E, 1)
        ok = (b > a) & (t[b, k] >= t_from) & (om[a, b] > 1) & (om[a, k] > 1) & (om[b, k] > 1)
        b, k = b[ok], k[ok]
        tt, x, y, z = t[b, k], om[a, b], om[b, k], om[a, k]
        cap = tt + theta + 1
        own = np.sort(np.stack([np.minimum(size[a] - x - z + tt, cap),
                                np.minimum(size[b] - x - y + tt, cap),
                                np.minimum(size[k] - y - z + tt, cap)], 1), 1)
        pair = np.sort(np.stack([x, y, z], 1), 1)
        for row in np.unique(np.concatenate([tt[:, None], pair, own], 1), axis=0):
            keys.add(tuple(row.tolist()))
    return len(keys)


WIDE = (70, 170, 12, 60, 31)


@pytest.mark.parametrize("theta", [1, 4])
def test_more_tuples_than_the_hash_holds(theta):
    """Level 3 tuples outside the table (5 common nodes or more) fill the hash
    of such tuples, and the rest goes straight to the histogram."""
    g = _wide(*WIDE)
    E = len(g[1]) - 1
    slots = 1 << 12
    while slots < E * (E - 1) / 4:      # at most this many: a quarter of the heavy entries
        slots *= 2
    assert _distinct_tuples(g, theta, 5) > slots
    h, h3 = _count(g, theta=theta)
    oh, o3 = oracle.count_exact(g[1], g[2], theta=theta)
    assert np.array_equal(h, oh) and np.array_equal(h3, o3)


def test_more_tuples_than_the_hash_holds_in_a_batch():
    gs = [_wide(*WIDE), _wide(12, 60, 2, 5, 32), _wide(70, 150, 12, 60, 33)]
    seeds = [4, 5, 6]
    _, _, _, _, ch, c3, _, _ = B.mochy_profile_batch(gs, 1, seeds)
    for g, (n, off, nodes) in enumerate(gs):
        o = oracle.profile(n, off, nodes, 1, seeds[g])
        assert np.array_equal(ch[g], o["counts_h"]) and np.array_equal(c3[g], o["counts_3h"])


def _popular(nodes, edges, popular, first, seed):
    """Hyperedges of 18 of `nodes` nodes, about alike in degree, and two of
    `popular` popular ones, whose ids come before (or after) all others."""
    rng = np.random.default_rng(seed)
    a, b = (popular, 0) if first else (0, nodes)
    sets = {tuple(sorted((rng.choice(nodes, 18, replace=False) + a).tolist() +
                         (rng.choice(popular, 2, replace=False) + b).tolist()))
            for _ in range(edges)}
    return (nodes + popular, *_util.csr_from_sets(sorted(sets)))


def _timed_count(g, **kw):
    with B.Context(**kw) as c:
        c.load(*g)
        c.project()
        got = c.count_exact()
        best = 1e9
        for _ in range(3):
            t = time.perf_counter()
            c.count_exact()
            best = min(best, time.perf_counter() - t)
    return got, best


def test_hubs_do_not_depend_on_the_order_of_ids():
    """More nodes of degree 32 or more than the hub matrix holds (4,096): the
    most popular are hubs whatever their ids.  As light nodes, a pair of them
    would cost the product of their degrees, some 5,000 each, on one warp."""
    last = _popular(5000, 13000, 5, False, 41)
    deg = np.bincount(last[2], minlength=last[0])
    assert (deg >= 32).sum() > 4200 and (deg[5000:] > 3000).all()
    first = _popular(5000, 13000, 5, True, 41)
    got, t_last = _timed_count(last)
    ref, t_first = _timed_count(first)
    split = _count(last, rest_path=2)
    for a, b, c in zip(got, ref, split):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    assert t_last < 3 * t_first, (t_last, t_first)


def test_hubs_of_crowded_units_in_a_batch():
    gs = [_wide(40, 90, 2, 6, 51), _popular(5000, 13000, 5, False, 42), _wide(3000, 1500, 2, 5, 52),
          _popular(4900, 12500, 3, True, 43)]
    seeds = [1, 2, 3, 4]
    cfg = B.mochy_config_default()
    cfg.rest_path = 2                    # the split kernels
    got = B.mochy_profile_batch(gs, 1, seeds)
    ref = B.mochy_profile_batch(gs, 1, seeds, cfg)
    assert np.array_equal(got[4], ref[4]) and np.array_equal(got[5], ref[5])


def _communities(edges, group, size, mult, seed):
    """`edges` hyperedges within communities of `group` nodes, mult * group
    drawn in each: nearly every one shares two nodes with some others, and
    line-graph rows are short."""
    rng = np.random.default_rng(seed)
    g = rng.integers(0, max(1, edges // (mult * group)), int(edges * 1.1) + 10)
    m = np.sort(g[:, None] * group + rng.integers(0, group, (len(g), size)), 1)
    m = np.unique(m[(np.diff(m, axis=1) > 0).all(1)], axis=0)
    m = m[rng.permutation(len(m))[:edges]]
    n = (max(1, edges // (mult * group))) * group
    return n, np.arange(len(m) + 1, dtype=np.int64) * size, m.astype(np.int32).ravel()


def _route(g, **kw):
    """Counts, and whether the levels made them."""
    with B.Context(**kw) as c:
        c.load(*g)
        c.project()
        B.mochy_trace(c.h, 1)
        got = c.count_exact()
        return got, "level 3" in B.mochy_trace_read(c.h)["phases_ms"]


@pytest.mark.parametrize("g,theta,levels", [
    ((110000, 50, 4, 3, 61), 1, False),      # sparse rows: an overlap matrix of 5 GB for few pairs
    ((6000, 1000, 10, 6, 62), 1, True),      # longer rows
    ((6000, 1000, 3, 6, 63), 3, True),
])
def test_sparse_hypergraphs_are_left_to_the_split_kernels(g, theta, levels):
    g = _communities(*g)
    (h, h3), by_levels = _route(g, theta=theta)
    oh, o3 = _count(g, theta=theta, rest_path=2)      # the split kernels
    assert np.array_equal(h, oh) and np.array_equal(h3, o3)
    assert by_levels == levels


@pytest.mark.parametrize("units,nodes,edges,most,levels", [(300, 200, 50, 12, False),
                                                           (12, 900, 900, 6, True)])
def test_batches_of_small_hypergraphs_are_left_to_the_split_kernels(units, nodes, edges, most,
                                                                     levels):
    kinds = [_wide(nodes, edges, 2, most, 700 + q) for q in range(4)]
    gs = [kinds[q % 4] for q in range(units)]
    seeds = list(range(units))
    _, _, _, _, ch, c3, _, info = B.mochy_profile_batch(gs, 3, seeds)
    for g in range(4):
        o = oracle.profile(*gs[g], 3, seeds[g])
        assert np.array_equal(ch[g], o["counts_h"]) and np.array_equal(c3[g], o["counts_3h"])
    assert (info["dense_threshold"] == 0) == levels


@pytest.mark.parametrize("theta", [1, 4])
def test_kh_motifs_of_a_sparse_hypergraph(theta):
    """k = 3 is the 3h-motifs, whichever of levels, scan and split counts."""
    g = _communities(110000, 50, 4, 3, 64)
    with B.Context(theta=theta) as c:
        c.load(*g)
        c.project()
        h, h3 = c.count_exact()
        kh, k3 = c.count_kh(3, (theta,))
    assert np.array_equal(h, kh) and np.array_equal(h3, k3)


def _groups(shared, own, counts):
    """For each count a group of that many hyperedges with `shared` nodes in
    common and `own` of their own: count - 1 heavy pairs each; and hyperedges
    across the groups, of one node of each."""
    sets, n, firsts = [], 0, []
    for k in counts:
        base = tuple(range(n, n + shared))
        firsts.append(n)
        n += shared
        for _ in range(k):
            sets.append(base + tuple(range(n, n + own)))
            n += own
    sets += [tuple(firsts), tuple(f + shared for f in firsts), (firsts[0], firsts[-1])]
    return (n, *_util.csr_from_sets(sets))


def _heavy_degrees(g):
    n, off, nodes = g
    m = np.zeros((len(off) - 1, n), np.int32)
    for i in range(len(off) - 1):
        m[i, nodes[off[i]:off[i + 1]]] = 1
    om = m @ m.T
    np.fill_diagonal(om, 0)
    return (om >= 2).sum(1)


@pytest.mark.parametrize("theta", [1, 4])
@pytest.mark.parametrize("shared,own", [(2, 1), (3, 2), (30, 4)])
def test_rows_of_16_and_17_heavy_pairs(shared, own, theta):
    """Rows of up to 16 heavy pairs are counted pair by pair, longer ones by
    classes; hyperedges of more than 32 nodes have no node masks."""
    g = _groups(shared, own, (16, 17, 18, 33, 34))
    assert {15, 16, 17, 32, 33} <= set(_heavy_degrees(g).tolist())
    h, h3 = _count(g, theta=theta)
    oh, o3 = oracle.count_exact(g[1], g[2], theta=theta)
    assert np.array_equal(h, oh) and np.array_equal(h3, o3)


def test_rows_of_16_and_17_heavy_pairs_in_a_batch():
    gs = [_groups(s, o, c) for s, o, c in ((2, 1, (17, 18)), (3, 2, (16, 17, 18)), (30, 4, (18, 17)))]
    gs = [g for g in gs for _ in range(3)]
    seeds = list(range(len(gs)))
    _, _, _, _, ch, c3, _, info = B.mochy_profile_batch(gs, 1, seeds)
    assert info["dense_threshold"] == 0      # by levels
    for g, (n, off, nodes) in enumerate(gs):
        o = oracle.profile(n, off, nodes, 1, seeds[g])
        assert np.array_equal(ch[g], o["counts_h"]) and np.array_equal(c3[g], o["counts_3h"])


def test_batches_of_ordinary_hypergraphs_go_by_levels():
    """Overlap matrices of 70 MB an input, more than 256 MB together: each fits the
    caches."""
    gs = []
    for q in range(4):
        spec = synth.HypergraphSpec(6000, 12000, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=800 + q)
        gs.append((6000, *synth.generate(spec)))
    seeds = [1, 2, 3, 4]
    cfg = B.mochy_config_default()
    cfg.rest_path = 2                    # the split kernels
    got = B.mochy_profile_batch(gs, 3, seeds)
    ref = B.mochy_profile_batch(gs, 3, seeds, cfg)
    assert got[7]["dense_threshold"] == 0
    assert np.array_equal(got[4], ref[4]) and np.array_equal(got[5], ref[5])


def _popular_sets(n, e, weights, z, seed):
    """`e` distinct hyperedges of 0, 1, ... nodes with these weights, members by
    Zipf(z) popularity, drawn one after another, repeats dropped."""
    rng = np.random.default_rng(seed)
    w = np.asarray(weights, float)
    size = rng.choice(len(w), 2 * e, p=w / w.sum())
    pop = np.arange(1, n + 1.0) ** -z
    draw = np.searchsorted(np.cumsum(pop / pop.sum()), rng.random((2 * e, 4 * len(w)))).clip(max=n - 1)
    sets = {}
    for k, d in zip(size, draw):
        s = tuple(sorted(list(dict.fromkeys(d.tolist()))[:k]))
        if len(s) == k:
            sets[s] = None
    return (n, *_util.csr_from_sets(list(sets)[:e]))


def test_hash_of_tuples_holds_those_of_a_dense_hypergraph():
    """700 hyperedges of 6 to 16 of 70 nodes: about 280,000 distinct tuples outside
    the table.  With a hash that they overflow, levels took 4 times what the
    split kernels take; with room for them, a fraction of it."""
    g = _popular_sets(70, 700, [0] * 6 + [1] * 11, 1.2, 91)
    got, t = _timed_count(g, theta=4)
    ref, t_split = _timed_count(g, theta=4, rest_path=2)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    assert t < 1.5 * t_split, (t, t_split)
