"""MoCHy-A and MoCHy-A+ on long line-graph rows (the kernel that stages a row
and streams the other), against the oracle's raw counts and estimates: wide
hyperedges without node masks, overlaps past its tables, thresholds up to the
last it covers and past it, draws below and above the number that is grouped."""
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


GRAPHS = {
    "dense": lambda: _random(30, 700, 2, 7, 1),
    "wide": lambda: _random(80, 400, 20, 45, 2),
    "zipf": lambda: (700, *synth.generate(
        synth.HypergraphSpec(700, 1600, 2, 25, "powerlaw", 2.2, "zipf", 1.1, seed=3))),
}
_cache = {}


def _graph(name):
    if name not in _cache:
        _cache[name] = GRAPHS[name]()
    return _cache[name]


@pytest.mark.parametrize("theta", [1, 2, 4, 5, 6, 7])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_long_rows_match_oracle(name, theta):
    n, off, nodes = _graph(name)
    with B.Context(theta=theta) as c:
        c.load(n, off, nodes)
        nw, _ = c.project()
        assert 2 * nw >= 256 * (c.hypergraph()[1].size - 1)      # the rows are long
        for method, samples in ((B.MOCHY_A, 20), (B.MOCHY_A_PLUS, 700), (B.MOCHY_A_PLUS, 4500)):
            g = c.count_sampled(method, samples, 11)
            o = oracle.count_sampled(off, nodes, method, samples, 11, theta=theta)
            for a, b in zip(g, o):
                assert np.array_equal(a, b), (method, samples)
