"""What a server reserves and what a batch puts into a wave include the
structures of the exact count by levels (needs a GB300).
"""
import numpy as np
import pytest

from paper_2310_15668_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _communities(edges, seed, group=200, size=6, mult=3):
    """Hyperedges within communities: short line-graph rows, nearly all with
    some heavy pairs, so that the overlap matrix is larger than the line graph."""
    rng = np.random.default_rng(seed)
    g = rng.integers(0, edges // (mult * group), int(edges * 1.1) + 10)
    m = np.sort(g[:, None] * group + rng.integers(0, group, (len(g), size)), 1)
    m = np.unique(m[(np.diff(m, axis=1) > 0).all(1)], axis=0)
    m = m[rng.permutation(len(m))[:edges]]
    return (edges // (mult * group) * group, np.arange(len(m) + 1, dtype=np.int64) * size,
            m.astype(np.int32).ravel())


def _need(g):
    n, off, nodes = g
    deg = np.bincount(nodes, minlength=n).astype(np.float64)
    w = float((0.5 * deg * (deg - 1)).sum())
    return int(16.0 * w + 96.0 * (off.size - 1) + 48.0 * int(off[-1]) + 16.0 * n) + (1 << 20)


def _alone(g):
    with B.Context() as c:
        c.load(*g)
        c.project()
        B.mochy_trace(c.h, 1)
        got = c.count_exact()
        assert "level 3" in B.mochy_trace_read(c.h)["phases_ms"]
        return got, B.mochy_device_bytes(c.h)


@pytest.mark.parametrize("room", ["all", "need"])
def test_a_server_reserves_what_the_levels_take(room):
    """With room for them the reservation covers what a context of its own holds
    for the same calls; without, the request runs within what it needs."""
    g = _communities(20000, 1)
    (h, h3), held = _alone(g)
    need = _need(g)
    assert held > 4 * need
    with B.Server(n_slots=2, budget=1 << 33 if room == "all" else need + 4096) as srv:
        r = srv.poll(srv.submit(B.MOCHY_REQ_EXACT, *g), wait_ms=120000)
        peak = srv.stats()["peak_reserved_bytes"]
    assert r["status"] >= 0
    assert np.array_equal(r["counts_h"], h) and np.array_equal(r["counts_3h"], h3)
    assert peak >= held if room == "all" else peak <= need + 4096


def test_server_results_do_not_depend_on_the_room():
    g = _communities(6000, 2)
    need = _need(g)
    got = []
    for budget in (1 << 33, 2 * need + 4096):
        with B.Server(n_slots=2, budget=budget) as srv:
            ts = [srv.submit(B.MOCHY_REQ_PROFILE, *g, n_random=2, seed=3),
                  srv.submit(B.MOCHY_REQ_SAMPLED, *g, method=B.MOCHY_A, samples=400, seed=4),
                  srv.submit(B.MOCHY_REQ_SAMPLED, *g, method=B.MOCHY_A_PLUS, samples=9000, seed=5)]
            got.append([srv.poll(t, wait_ms=120000) for t in ts])
            assert srv.stats()["peak_reserved_bytes"] <= budget
    for a, b in zip(*got):
        assert a["status"] >= 0 and b["status"] >= 0
        for k in ("counts_h", "counts_3h", "est_3h", "cp_3h"):
            assert np.array_equal(a[k], b[k])


def test_waves_of_a_batch_leave_room_for_the_levels():
    gs = [_communities(5000, 10 + q) for q in range(6)]
    seeds = list(range(6))
    cfg = B.mochy_config_default()
    cfg.hbm_budget_bytes = int(1.05 * 3 * sum(_need(g) for g in gs))
    got = B.mochy_profile_batch(gs, 2, seeds, cfg)
    ref = B.mochy_profile_batch(gs, 2, seeds)
    assert ref[7]["n_waves"] == 1 and ref[7]["dense_threshold"] == 0      # by levels
    assert got[7]["n_waves"] > 1 and got[7]["dense_threshold"] == 0
    for a, b in zip(got[:7], ref[:7]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("theta", [0, -7])
def test_a_bad_theta_is_refused_as_ever(theta):
    cfg = B.mochy_config_default()
    cfg.theta = theta
    with pytest.raises(B.MochyError) as e:
        B.mochy_profile_batch([_communities(1000, 3)], 1, [1], cfg)
    assert e.value.code == B.E_INVALID
