"""The measured tuner's threshold is the one that the following counts take
(needs a GB300).
"""
import numpy as np
import pytest

import oracle
from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _traced(c):
    B.mochy_trace(c.h, 1)
    got = c.count_exact()
    t = B.mochy_trace_read(c.h)
    B.mochy_trace(c.h, 0)
    return got, t["dense_threshold"], "level 3" in t["phases_ms"]


@pytest.mark.parametrize("theta", [1, 5])
def test_counts_take_the_tuned_threshold(theta):
    spec = synth.HypergraphSpec(600, 1200, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=21)
    off, nodes = synth.generate(spec)
    with B.Context(theta=theta) as c:
        c.load(spec.n_nodes, off, nodes)
        c.project()
        ref, thr, by_levels = _traced(c)
        assert by_levels == (theta == 1) and (thr == 0) == by_levels
        before = c.profile(1, 3)
        best, _ = B.mochy_tune_dense_threshold(c.h, [48, 96], 0.2, 3)
        got, thr, by_levels = _traced(c)
        assert thr == best and not by_levels
        after = c.profile(1, 3)
        c.load(spec.n_nodes, off, nodes)      # the context's, not the line graph's
        c.project()
        again, thr, by_levels = _traced(c)
        assert thr == best and not by_levels
    o = oracle.count_exact(off, nodes, theta=theta)
    for r in (ref, got, again):
        assert np.array_equal(r[0], o[0]) and np.array_equal(r[1], o[1])
    assert np.array_equal(before["counts_3h"], after["counts_3h"])
