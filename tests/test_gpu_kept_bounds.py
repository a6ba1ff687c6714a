"""Bounds on the device memory that a context keeps after giving it up (needs a
GB300).
"""
import pytest

from paper_2310_15668_gb300 import binding as B, synth

pytestmark = pytest.mark.gpu

GB = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_a_context_and_its_copies_keep_16_gb_together():
    """The line graphs (about 9 GB each, the copy's too) and overlap matrices of a
    profile, kept when a small hypergraph takes their place."""
    spec = synth.HypergraphSpec(300, 100000, 6, 6, "uniform", 0.0, "uniform", 0.0, seed=31)
    off, nodes = synth.generate(spec)
    tiny = synth.generate(synth.TINY)
    with B.Server(n_slots=1) as srv:
        budget = srv.stats()["budget_bytes"]
    with B.Context() as warm:
        warm.load(synth.TINY.n_nodes, *tiny)
    before = _used()
    with B.Context() as c:
        c.load(spec.n_nodes, off, nodes)
        c.profile(1, 3)
        held = B.mochy_device_bytes(c.h)
        assert held > 8 * GB
        c.load(synth.TINY.n_nodes, *tiny)
        kept = _used() - before
        assert B.mochy_device_bytes(c.h) < GB
        assert 8 * GB < kept < 17.5 * GB
        # what is kept is there for a server or a batch
        with B.Server(n_slots=1) as srv:
            assert abs(srv.stats()["budget_bytes"] - budget) < 2 * GB
        c.profile(1, 3)
    assert _used() - before < GB
