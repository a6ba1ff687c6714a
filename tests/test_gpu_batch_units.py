"""Batches of more hypergraphs than one dimension of a grid but x takes (needs
a GB300), against the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2310_15668_gb300 import binding as B
from . import _util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_more_than_65535_units_in_one_wave():
    graphs, copies = 2200, 31
    kinds = [_util.micro_graph(500 + q, n_nodes=8, n_edges=6 + q % 7, s_max=5) for q in range(20)]
    gs = [(8, *_util.csr_from_sets(kinds[g % len(kinds)])) for g in range(graphs)]
    seeds = [70 + g for g in range(graphs)]
    _, _, _, _, ch, c3, _, info = B.mochy_profile_batch(gs, copies, seeds)
    assert info["n_units"] == graphs * (copies + 1) > 65536 and info["n_waves"] == 1
    for g in (0, 1, 1023, 2046, 2047, 2048, 2049, graphs - 1):   # units 65,535 and 65,536: 2,047 and 2,048
        o = oracle.profile(*gs[g], copies, seeds[g])
        assert np.array_equal(ch[g], o["counts_h"]) and np.array_equal(c3[g], o["counts_3h"])
    # the inputs of one kind count the same
    assert (c3[:, 0].reshape(-1, len(kinds), 431) == c3[:len(kinds), 0]).all()
