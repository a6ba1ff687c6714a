"""The work that users of this library have it do, as measurable cases.

Every case is one call sequence through the public entry points of
``paper_2310_15668_gb300.binding`` on a seeded hypergraph of the shapes that
the library's own workloads have (``synth.py``, ``bench.py``): hyperedge
sizes from a truncated power law on [2, 25] or uniform on [2, 5], members by
Zipf or uniform node popularity, N = E / 2 nodes.  Hypergraphs are drawn on
the GPU and handed over as host arrays, as a program that has read a dataset
holds them; the context is the handle such a program keeps.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2310_15668_gb300 import binding as B

# Kinds of case:
#   count    load a hypergraph, project it, count every h- and 3h-motif exactly
#   project  load a hypergraph and build its line graph, degrees read back
#   sample   MoCHy-A / MoCHy-A+ estimates on a projected hypergraph
#   otf      load a hypergraph, MoCHy-A+ estimates without its line graph
#   profile  load a hypergraph, significance and characteristic profile
#   batch    the profiles of several hypergraphs in one call
#   kh       kh-motif counts of a projected hypergraph


def _zipf(name, kind, edges, z=1.0, alpha=2.5, **more):
    return dict(name=name, kind=kind, edges=edges, nodes=max(edges // 2, 64), law="zipf", z=z,
                alpha=alpha, s_min=2, s_max=25, theta=1, **more)


def listed():
    return [
        # the smallest exact count (the benchmark's tiny configuration): a
        # sparse hypergraph, where launches and host work count
        dict(name="count-tiny", kind="count", edges=2000, nodes=1000, law="uniform", z=0.0,
             alpha=0.0, s_min=2, s_max=5, theta=1),
        # an ordinary request of the serving workload (E in [1,000, 4,000])
        _zipf("count-2k", "count", 2003),
        # an ordinary dataset (the paper's contact and e-mail hypergraphs)
        _zipf("count-10k", "count", 10000),
        # a large exact count on a hub-dominated line graph
        _zipf("count-60k", "count", 60000),
        # 3h-motifs with another threshold (theta = 2)
        dict(_zipf("count-theta2", "count", 7001), theta=2),
        # a line graph of hundreds of millions of hyperwedges
        _zipf("project-100k", "project", 100001),
        # hyperwedge sampling on a projected hypergraph
        _zipf("sample-aplus", "sample", 100000, method="A+", samples=200000),
        # hyperedge sampling on a projected hypergraph
        _zipf("sample-a", "sample", 30011, method="A", samples=500),
        # hyperwedge sampling where the line graph would not fit (the
        # benchmark's large configuration, scaled)
        _zipf("otf-500k", "otf", 500000, z=1.1, alpha=2.2, samples=20000),
        # a characteristic profile, one hypergraph at a time (serving mix)
        _zipf("profile-2k", "profile", 2000, copies=4),
        # characteristic profiles of several hypergraphs in one call
        _zipf("batch-6", "batch", 2000, graphs=6, copies=8),
        # 4h-motifs of an ordinary hypergraph
        _zipf("kh4-4k", "kh", 4001, k=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "count", "project", "sample", "sample", "otf", "profile",
                       "batch", "kh"])
    z, alpha = rng.uniform(0.8, 1.0), rng.uniform(2.4, 2.8)
    if kind == "count":
        theta = rng.choice([1, 1, 2])
        if rng.random() < 0.25:   # uniform members, small hyperedges
            e = _log(rng, 1000, 60000)
            return dict(kind=kind, edges=e, nodes=max(e // 2, 64), law="uniform", z=0.0,
                        alpha=0.0, s_min=2, s_max=rng.choice([4, 5, 8]), theta=theta)
        c = _zipf("", kind, _log(rng, 500, 40000 if theta == 1 else 7000), z, alpha)
        c["theta"] = theta
    elif kind == "project":
        c = _zipf("", kind, _log(rng, 5000, 100000), z, alpha)
    elif kind == "sample":
        if rng.random() < 0.6:
            c = _zipf("", kind, _log(rng, 5000, 100000), z, alpha, method="A+",
                      samples=_log(rng, 5000, 200000))
        else:
            c = _zipf("", kind, _log(rng, 3000, 30000), z, alpha, method="A",
                      samples=_log(rng, 50, 500))
    elif kind == "otf":
        c = _zipf("", kind, _log(rng, 50000, 500000), rng.uniform(0.9, 1.1),
                  rng.uniform(2.2, 2.6), samples=_log(rng, 1000, 20000))
    elif kind == "profile":
        c = _zipf("", kind, _log(rng, 300, 2000), z, alpha, copies=rng.randint(1, 4))
    elif kind == "batch":
        c = _zipf("", kind, _log(rng, 300, 2000), z, alpha, graphs=rng.randint(2, 6),
                  copies=rng.randint(2, 8))
    else:
        c = _zipf("", kind, _log(rng, 500, 4000), z, alpha, k=rng.choice([2, 3, 4]))
    c.pop("name")
    return c


def _size_weights(case):
    s = np.arange(case["s_min"], case["s_max"] + 1, dtype=np.float64)
    w = np.ones_like(s) if case["alpha"] == 0.0 else s ** -case["alpha"]
    return s, w / w.sum()


def _node_weights(case, n_nodes):
    w = np.ones(n_nodes) if case["law"] == "uniform" else \
        np.arange(1, n_nodes + 1, dtype=np.float64) ** -case["z"]
    return w / w.sum()


def _candidates(case, n, nodes, scdf, ncdf, gen):
    """n candidate hyperedges, members ascending in rows padded with -1."""
    dev = scdf.device
    u = torch.rand(n, device=dev, dtype=torch.float64, generator=gen)
    size = case["s_min"] + torch.searchsorted(scdf, u, right=True).clamp_(max=len(scdf) - 1)
    u = torch.rand(n, 2 * case["s_max"] + 8, device=dev, dtype=torch.float64, generator=gen)
    d = torch.searchsorted(ncdf, u, right=True).clamp_(max=nodes - 1)
    # the first occurrence of each member, in draw order
    key, order = torch.sort(d, dim=1, stable=True)
    first = torch.ones_like(key, dtype=torch.bool)
    first[:, 1:] = key[:, 1:] != key[:, :-1]
    keep = torch.zeros_like(first).scatter_(1, order, first)
    keep &= keep.cumsum(1) <= size[:, None]
    m = torch.sort(torch.where(keep, d, torch.full_like(d, 1 << 40)), dim=1)[0]
    m = m[:, :case["s_max"]]
    return torch.where(m < (1 << 40), m, torch.full_like(m, -1))


def _hypergraph(case, edges, nodes, seed):
    """(offsets int64, nodes int32) host arrays of `edges` distinct hyperedges:
    sizes by the case's law, members drawn one after another, repeats redrawn
    (a row that runs out of draws keeps the members that it has)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    scdf = torch.tensor(np.cumsum(_size_weights(case)[1]), device=dev)
    ncdf = torch.tensor(np.cumsum(_node_weights(case, nodes)), device=dev)
    mult = torch.randint(-(1 << 62), 1 << 62, (case["s_max"],), dtype=torch.int64, device=dev,
                         generator=gen) | 1
    rows = torch.empty(0, case["s_max"], dtype=torch.int64, device=dev)
    while len(rows) < edges:
        n = max(1024, min(1 << 18, int(1.3 * (edges - len(rows)))))
        rows = torch.cat([rows, _candidates(case, n, nodes, scdf, ncdf, gen)])
        # the first row of each member set, by a 64-bit product sum of its members
        v = rows + 2
        h, order = torch.sort((v * v * v * mult + (v ^ (v << 17)) * mult.flip(0)).sum(1),
                              stable=True)
        new = torch.ones_like(h, dtype=torch.bool)
        new[1:] = h[1:] != h[:-1]
        rows = rows[torch.sort(order[new])[0]]
    rows = rows[:edges]
    off = torch.zeros(edges + 1, dtype=torch.int64, device=dev)
    off[1:] = torch.cumsum((rows >= 0).sum(1), 0)
    return off.cpu().numpy(), rows[rows >= 0].to(torch.int32).cpu().numpy()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "batch":
        # hyperedge counts spread over a factor of ten, as a collection's are
        st["graphs"] = []
        for g in range(case["graphs"]):
            e = int(case["edges"] * 10.0 ** (-g / max(case["graphs"] - 1, 1)))
            n = max(e // 2, 64)
            st["graphs"].append((n, *_hypergraph(case, e, n, seed * 1000003 + g)))
        return st
    st["off"], st["nodes"] = _hypergraph(case, case["edges"], case["nodes"], seed)
    st["ctx"] = B.Context(theta=case["theta"])
    if kind in ("sample", "kh"):
        st["ctx"].load(case["nodes"], st["off"], st["nodes"])
        st["ctx"].project()
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "batch":
        sig_h, cp_h, sig_3h, cp_3h, ch, c3, _, _ = B.mochy_profile_batch(
            st["graphs"], case["copies"], [st["seed"] + g for g in range(case["graphs"])])
        return dict(sig_h=sig_h, cp_h=cp_h, sig_3h=sig_3h, cp_3h=cp_3h, counts_h=ch, counts_3h=c3)
    c = st["ctx"]
    if kind == "sample":
        method = B.MOCHY_A_PLUS if case["method"] == "A+" else B.MOCHY_A
        return c.count_sampled(method, case["samples"], st["seed"])
    if kind == "kh":
        return c.count_kh(case["k"], (1, 2)[:case["k"] - 2])
    c.load(case["nodes"], st["off"], st["nodes"])
    if kind == "count":
        n_wedges, max_degree = c.project()
        return (n_wedges, max_degree) + tuple(c.count_exact())
    if kind == "project":
        n_wedges, max_degree = c.project()
        return n_wedges, max_degree, c.line_degrees()
    if kind == "otf":
        return c.count_sampled_onthefly(case["samples"], st["seed"])
    p = c.profile(case["copies"], st["seed"])
    return {k: p[k] for k in ("sig_h", "cp_h", "sig_3h", "cp_3h", "counts_h", "counts_3h")}


def _expected(case, edges, nodes):
    """Expected incidences and hyperwedges of one hypergraph of the case."""
    s, w = _size_weights(case)
    p = _node_weights(case, nodes)
    mean = float((s * w).sum())
    # members of a hyperedge of the mean size, by node
    inc = 1.0 - np.exp(-mean * p)
    share = 1.0 - math.exp(-float((inc * inc).sum()))
    return edges * mean, 0.5 * edges * edges * share


def work(case):
    """Bytes: the hypergraph read once, the line graph (16 bytes a hyperwedge)
    written once where the calls build one and read once where they count on
    it, the results written once; for samples, the rows of each draw read
    once.  Operations: one per result value (the counts need no more than
    sums over what is read)."""
    kind = case["kind"]
    inc, wedges = _expected(case, case["edges"], case["nodes"])
    graph = 4 * inc + 8 * case["edges"]
    degree = 2.0 * wedges / case["edges"]
    counts = 457 * 8
    if kind == "count":
        return dict(bytes=graph + 32 * wedges + counts, flops=457)
    if kind == "project":
        return dict(bytes=graph + 16 * wedges + 8 * case["edges"], flops=case["edges"])
    if kind == "kh":
        return dict(bytes=16 * wedges + 3102 * 8, flops=3102)
    if kind == "sample":
        rows = 2 * degree if case["method"] == "A+" else degree * degree
        return dict(bytes=case["samples"] * rows * 8 + 2 * counts, flops=914)
    if kind == "otf":
        # bitmaps of the most popular nodes: E / 8 bytes for each, over the
        # few nodes of a drawn hyperwedge
        return dict(bytes=graph + case["samples"] * case["edges"] / 8 + 2 * counts, flops=914)
    total = flops = 0.0
    for g in range(case.get("graphs", 1)):
        e = case["edges"] if kind == "profile" else \
            int(case["edges"] * 10.0 ** (-g / max(case["graphs"] - 1, 1)))
        i, v = _expected(case, e, max(e // 2, 64))
        total += (1 + case["copies"]) * (4 * i + 8 * e + 32 * v + counts) + 4 * counts
        flops += 914 * (1 + case["copies"])
    return dict(bytes=total, flops=flops)


def _distinct(off, nodes):
    """Member sets of the distinct hyperedges, first occurrences in order."""
    return list(dict.fromkeys(tuple(nodes[off[i]:off[i + 1]].tolist())
                              for i in range(len(off) - 1)))


def _incidence(edges, n_nodes, dtype):
    rows = np.repeat(np.arange(len(edges)), [len(e) for e in edges])
    x = torch.zeros(len(edges), n_nodes, dtype=dtype, device="cuda")
    x[torch.from_numpy(rows).cuda(), torch.tensor([v for e in edges for v in e]).cuda()] = 1
    return x


def _motif_table():
    """3h-motif id of each ternary region code (regions (1) to (7)), the
    h-motif of each 3h-motif: patterns of three distinct, connected
    hyperedges up to their order, numbered as the library's header states."""
    pairs = {(0, 1): 3, (1, 2): 4, (0, 2): 5}
    perm = []
    for o in itertools.permutations(range(3)):
        perm.append(list(o) + [pairs[tuple(sorted((o[a], o[b])))] for a, b in pairs] + [6])
    member = [(0, 3, 5, 6), (1, 3, 4, 6), (2, 4, 5, 6)]

    def valid(c):
        sets = [tuple(c[r] > 0 for r in range(7) if (r in member[e])) for e in range(3)]
        if not all(any(s) for s in sets):
            return False
        adj = [c[pairs[p]] > 0 or c[6] > 0 for p in pairs]
        if sum(adj) < 2:
            return False
        # two hyperedges with no region of their own would be the same set
        for a, b in pairs:
            only = [r for r in range(7) if (r in member[a]) != (r in member[b])]
            if not any(c[r] for r in only):
                return False
        return True

    def canonical(c):
        return min(tuple(c[q] for q in p) for p in perm)

    def group(c):
        if c[6]:
            return 0
        adj = sum(c[pairs[p]] > 0 for p in pairs)
        return 1 if adj == 2 else 2

    two = sorted({canonical(c) for c in itertools.product((0, 1), repeat=7) if valid(c)},
                 key=lambda c: (group(c), c))
    h_of = {c: i + 1 for i, c in enumerate(two)}
    parent = {}
    for c in itertools.product((0, 1, 2), repeat=7):
        if valid(c):
            k = canonical(c)
            parent[k] = h_of[canonical(tuple(int(v > 0) for v in k))]
    three = sorted(parent, key=lambda c: (parent[c], c))
    id_of = {c: i + 1 for i, c in enumerate(three)}
    lut = np.zeros(3 ** 7, np.int64)
    for c in itertools.product((0, 1, 2), repeat=7):
        if valid(c):
            lut[sum(v * 3 ** r for r, v in enumerate(c))] = id_of[canonical(c)]
    return lut, np.array([0] + [parent[c] for c in three])


def _exact_count(case, edges, n_wedges, max_degree):
    x = _incidence(edges, case["nodes"], torch.float64)
    om = (x @ x.T).round().to(torch.int64)
    size = om.diagonal().clone()
    om.fill_diagonal_(0)
    lut, parent = _motif_table()
    lut = torch.from_numpy(lut).cuda()
    h3 = torch.zeros(432, dtype=torch.int64, device="cuda")
    adj = om > 0
    for i in range(len(edges)):
        nb = torch.nonzero(adj[i]).ravel()
        if len(nb) < 2:
            continue
        p, q = torch.triu_indices(len(nb), len(nb), 1, device="cuda")
        j, k = nb[p], nb[q]
        w = om[j, k]
        ok = (w == 0) | (i < j)   # open: at its centre; closed: at its smallest
        j, k, w = j[ok], k[ok], w[ok]
        inside = x[nb] * x[i]
        t = (inside @ inside.T).round().to(torch.int64)[p[ok], q[ok]]
        a, b = om[i, j], om[i, k]
        reg = (size[i] - a - b + t, size[j] - a - w + t, size[k] - w - b + t, a - t, w - t, b - t,
               t)
        code = sum(((r > 0).long() + (r > case["theta"]).long()) * 3 ** s
                   for s, r in enumerate(reg))
        h3 += torch.bincount(lut[code], minlength=432)
    c3 = h3.cpu().numpy()[1:]
    h = np.bincount(parent[1:], weights=c3, minlength=27)[1:].astype(np.int64)
    return n_wedges, max_degree, h, c3


def exact(case, seed):
    """Line-graph degrees by dense products of incidence rows, and for small
    sparse hypergraphs the motif counts by going over every pair of
    neighbours of every hyperedge.  The other outputs have no value that can
    be had in seconds without the library (the estimates and profiles belong
    to its random draws)."""
    small = case["kind"] == "count" and case["law"] == "uniform" and case["edges"] <= 3000
    if not small and case["kind"] != "project":
        return None
    edges = _distinct(*_hypergraph(case, case["edges"], case["nodes"], seed))
    x = _incidence(edges, case["nodes"], torch.float16)   # sums of ones: exact
    deg = torch.cat([((x[i:i + 4096] @ x.T) > 0).sum(1) - 1 for i in range(0, len(edges), 4096)])
    del x
    n_wedges, max_degree = int(deg.sum()) // 2, int(deg.max())
    if small:
        return _exact_count(case, edges, n_wedges, max_degree)
    return n_wedges, max_degree, deg.cpu().numpy()
