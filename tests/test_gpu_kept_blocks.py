"""Device blocks kept between calls (needs a GB300): one context that loads,
projects, counts, samples and profiles hypergraphs of growing and shrinking
sizes gives what a fresh context gives each time, also within a budget that
refuses one of them and beside contexts on other threads.
"""
import threading

import numpy as np
import pytest

from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu

SPECS = [synth.HypergraphSpec(max(e // 2, 500), e, 2, 25, "powerlaw", 2.5, "zipf", 1.0, seed=e)
         for e in (300, 5000, 4100, 64, 5200, 1000)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _all(c, spec):
    off, nodes = synth.generate(spec)
    c.load(spec.n_nodes, off, nodes)
    fly = c.count_sampled_onthefly(50, 3)
    out = [*c.project(), *c.count_exact(), *c.count_sampled(B.MOCHY_A_PLUS, 50, 3), *fly[:4]]
    p = c.profile(2, 7)
    return out + [p[k] for k in ("sig_h", "cp_h", "sig_3h", "cp_3h", "counts_h", "counts_3h")]


def _same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def _fresh():
    out = []
    for s in SPECS:
        with B.Context() as c:
            out.append(_all(c, s))
    return out


def test_one_context_for_many_sizes():
    ref = _fresh()
    with B.Context() as c:
        for _ in range(2):
            for s, r in zip(SPECS, ref):
                _same(_all(c, s), r)


def test_within_a_budget():
    """A context whose budget refuses one size serves the others before and
    after, and never holds more than the budget."""
    ref = _fresh()
    big = max(range(len(SPECS)), key=lambda q: SPECS[q].n_edges)
    off, nodes = synth.generate(SPECS[big])
    with B.Context() as c:
        c.load(SPECS[big].n_nodes, off, nodes)
        line_graph = 16 * c.project()[0]
    with B.Context(budget=line_graph) as c:
        for _ in range(2):
            for q in (0, big, 3, 5):
                if q == big:
                    with pytest.raises(B.MochyError) as e:
                        _all(c, SPECS[q])
                    assert e.value.code == B.E_NOMEM
                else:
                    _same(_all(c, SPECS[q]), ref[q])
                assert B.mochy_device_bytes(c.h) <= line_graph


def test_contexts_on_threads():
    ref = _fresh()
    bad = []

    def work(k):
        try:
            with B.Context() as c:
                for q in range(len(SPECS)):
                    s = (q + k) % len(SPECS)
                    _same(_all(c, SPECS[s]), ref[s])
        except Exception as e:      # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
