"""Least device memory budgets (needs a GB300): memory that a call could do
without does not make it, or the calls after it, fail where they fitted.
"""
import numpy as np
import pytest

from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu

SPEC = synth.HypergraphSpec(2000, 4001, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=77)
FLAT = synth.HypergraphSpec(3000, 6001, 2, 5, "uniform", 0.0, "uniform", 0.0, seed=78)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _graph(spec):
    return (spec.n_nodes, *synth.generate(spec))


def _fits(budget, calls, **kw):
    """What the calls return within the budget, or None when it refuses one."""
    try:
        with B.Context(budget=budget, **kw) as c:
            out = [f(c) for f in calls]
            assert B.mochy_device_bytes(c.h) <= budget
            return out
    except B.MochyError as e:
        assert e.code == B.E_NOMEM
        return None


def _least(calls, lo=1 << 16, hi=1 << 32, **kw):
    """Least budget, to 256 bytes, and what the calls return with it."""
    got = _fits(hi, calls, **kw)
    assert got is not None
    while hi - lo > 256:
        mid = (lo + hi) // 2
        r = _fits(mid, calls, **kw)
        if r is None:
            lo = mid
        else:
            hi, got = mid, r
    return hi, got


def _load(g):
    return lambda c: c.load(*g)


def _project(c):
    return c.project()[0], c.line_degrees()


@pytest.mark.parametrize("spec", [SPEC, FLAT])
def test_projection_needs_the_line_graph_alone(spec):
    """Beside what a load leaves: three offset arrays, one word a hyperedge and
    the line graph's entries."""
    g = _graph(spec)
    E = len(g[1]) - 1
    with B.Context() as c:
        c.load(*g)
        loaded = B.mochy_device_bytes(c.h)
        nw, deg = _project(c)
    need = loaded + 8 * (3 * E + 2) + 4 * E + 16 * nw
    got = _fits(need + 64, [_load(g), _project])
    assert got is not None
    assert got[1][0] == nw and np.array_equal(got[1][1], deg)
    # the rows themselves: the same draws and counts
    calls = [_load(g), _project, lambda c: c.count_sampled(B.MOCHY_A_PLUS, 300, 5)]
    for a, b in zip(_fits(need + (1 << 20), calls)[2], _fits(1 << 32, calls)[2]):
        assert np.array_equal(a, b)


def _exact(c):
    return c.count_exact()


def _profiles(c):
    return c.hyperedge_profile()


@pytest.mark.parametrize("spec", [SPEC, FLAT])
@pytest.mark.parametrize("after", [(), (_profiles,), (lambda c: c.count_kh(2, ()),)])
def test_exact_counts_fit_where_the_split_kernels_do(spec, after):
    """The level structures are taken where there is room for them, and given
    up for a later call that needs it."""
    calls = [_load(_graph(spec)), _project, _exact, *after]
    with_levels, got = _least(calls)
    split, ref = _least(calls, rest_path=2)
    assert with_levels <= split
    for a, b in zip(got[2:], ref[2:]):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


def test_sampling_leaves_its_room_to_later_calls():
    """Class histograms and grouped draws of long rows are scratch of the call."""
    g = _graph(SPEC)
    assert 2 * 1462159 >= 256 * (len(g[1]) - 1)          # long enough rows for both methods
    samples = [lambda c: c.count_sampled(B.MOCHY_A, 300, 3),
               lambda c: c.count_sampled(B.MOCHY_A_PLUS, 9000, 4)]
    without, _ = _least([_load(g), _project, _profiles])
    sampled, got = _least([_load(g), _project, *samples, _profiles])
    assert sampled <= without
    for a, b in zip(got[2:4], _fits(1 << 32, [_load(g), _project, *samples])[2:]):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
