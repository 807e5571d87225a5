"""Sizes at which the CUDA kernels change form, each against the oracle on the
same input (whole numbers: equal, no tolerance):

- hyperedge lengths at the edges of the segment kernels' buckets (pin counts,
  contraction);
- incidence counts at the edge between a block's flattened and grouped visit,
  in hash tables and in arrays, sums that fit one word and sums that do not in
  one launch;
- vertex counts at the edges of the key spaces that arrays hold;
- numbers of heavy vertices at the edges of the array tier's forms;
- connection rows that run out of room on the way to the finest level;
- two hyperedges of different content under one 64-bit key.
"""
import numpy as np
import pytest
import torch

import oracle
import snngen
from gpu_helpers import lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as g
    g.build()
    import paper_2609_07577_gb300 as P
    P.lib()
    assert torch.cuda.is_available()


def _net(name, V, hedges, w, omega, delta, phi):
    """hedges: (source, destinations) pairs."""
    pins, off = [], [0]
    for s, d in hedges:
        d = np.unique(np.asarray(d))
        pins.append(np.concatenate([[s], d[d != s]]))
        off.append(off[-1] + pins[-1].size)
    return snngen.Hypergraph(name, V, np.asarray(off, np.int64), np.concatenate(pins).astype(np.int32),
                             np.asarray(w, np.int32), omega, delta, phi)


def _same_pass(hg, rows=None, setup=None):
    from paper_2609_07577_gb300 import HGraph, params_for
    rho_o, cost_o, st_o, _, _ = oracle.partition(hg, oracle.params_of(hg))
    G = HGraph.from_hypergraph(hg, params=params_for(hg.omega, hg.delta, hg.phi))
    try:
        if rows is not None:
            G.set_row_budget(rows)
        if setup is not None:
            setup(G)
        rho, cost, st = G.partition()
        logs = G.round_logs()
    finally:
        G.close()
    assert cost == cost_o and np.array_equal(rho.cpu().numpy(), rho_o)
    assert st["rounds"] == st_o["rounds"] and st["moves"] == st_o["moves"]
    return logs


@pytest.mark.parametrize("rows", [0, None])
def test_segment_lengths(rows):
    rng = np.random.default_rng(1)
    V, hedges = 3000, []
    for n in (2, 3, 4, 5, 31, 32, 33, 34, 63, 64, 65, 66, 127, 128, 129, 130, 255, 256, 257, 258, 1023,
              1024, 1025, 2100):
        for _ in range(3):   # n pins: the source and n - 1 destinations
            p = rng.choice(V, n, replace=False)
            hedges.append((p[0], p[1:]))
    hg = _net("lengths", V, hedges, rng.integers(1, 9, len(hedges)), 200, 4000, 100000)
    assert lockstep(hg, max_levels=3) >= 2
    _same_pass(hg, rows)


# hubs of exactly these incidence counts: the flattened form takes up to a
# quarter of a block's threads, 64 in the block and 128 in the big tier
HUBS = [63, 64, 65, 66, 127, 128, 129, 130, 300]


@pytest.mark.parametrize("wmax", [1, 1 << 22], ids=["packed", "mixed"])
@pytest.mark.parametrize("zero", [False, True], ids=["arrays", "tables"])
@pytest.mark.parametrize("tiers", [None, (0, 1 << 40, 1 << 40), (0, 0, 1 << 40)],
                         ids=["rule", "block", "big"])
def test_incidence_counts(tiers, zero, wmax):
    rng = np.random.default_rng(2)
    V, hedges, w = 5200, [], []
    for h, deg in enumerate(HUBS * 2):
        for i in range(deg):
            d = rng.choice(np.arange(1100, V), 24, replace=False)
            hedges.append((2 * len(HUBS) + int(rng.integers(1000)), np.append(d, h)))
            # sums of the second half's hubs pass 32 bits only with large weights
            w.append(int(rng.integers(1, 4)) * (wmax if h >= len(HUBS) else 1))
    if zero:
        w[0] = 0   # presence is no longer a nonzero sum: tables on every level
    hg = _net("hubs", V, hedges, w, 64, 1 << 20, 1 << 20)

    def setup(G):
        G.set_coarsen_mode(1)
        G.set_row_budget(0)
        if tiers:
            G.set_histogram_tiers(*tiers)
    assert lockstep(hg, max_levels=2, setup=setup) == 2


@pytest.mark.parametrize("V", [4095, 4096, 4097, 24575, 24576, 24577])
def test_key_spaces(V):
    rng = np.random.default_rng(V)
    hedges = [(int(s), rng.choice(V, 6, replace=False)) for s in rng.choice(V, V // 4, replace=False)]
    hedges += [(int(s), np.append(rng.choice(V, 400, replace=False), [0, V - 1])) for s in (1, 2, V - 2)]
    hg = _net("keys", V, hedges, rng.integers(1, 5, len(hedges)), 40, 1000, 5000)
    for budget in (0, None):
        assert lockstep(hg, max_levels=2,
                        setup=lambda G: G.set_row_budget(0) if budget == 0 else None) == 2


@pytest.mark.parametrize("heavy", [1, 37, 38, 39, 303, 304, 305])
def test_heavy_vertex_counts(heavy):
    """`heavy` vertices meet more keys than a warp's table holds; the rest
    stay in the warp tier. Both by the rule and as the big tier's."""
    rng = np.random.default_rng(heavy)
    V = 6000
    p = rng.permutation(V)
    hedges = [(p[0], p[1:heavy]), (p[heavy + 1], np.concatenate([p[:heavy], p[heavy + 2:384]])),
              (p[400], np.concatenate([p[:heavy], p[401:401 + 383 - heavy]]))]
    hedges = [h for h in hedges if len(h[1])]
    hg = _net("heavy", V, hedges, [3] * len(hedges), 50, 1000, 5000)
    for tiers in (None, (0, 0, 1 << 40)):
        def setup(G):
            G.set_coarsen_mode(1)
            G.set_row_budget(0)
            if tiers:
                G.set_histogram_tiers(*tiers)
        assert lockstep(hg, max_levels=2, setup=setup) >= 1


@pytest.mark.parametrize("name", ["cfg1", "cfg2s"])
@pytest.mark.parametrize("share", [0.02, 0.3, 0.6, 0.95])
def test_rows_out_of_room(name, share):
    """Coarse levels have connection rows, finer ones find no room."""
    hg = snngen.by_name(name)
    K = oracle.partition(hg, oracle.params_of(hg))[2]["n_parts"]
    _same_pass(hg, rows=int(share * 8 * ((K + 3) // 4 * 4) * hg.V))


def _mix64(x):
    """csrc/common.cuh mix64"""
    x = x.astype(np.uint64) + np.uint64(0x9e3779b97f4a7c15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
    return x ^ (x >> np.uint64(31))


def _join(a, b, ia, ib, bits, shift):
    """Pairs of a and b whose sums are 0 in `bits` bits from `shift`."""
    m = np.uint64((1 << bits) - 1)
    ka = (a >> np.uint64(shift)) & m
    kb = (np.uint64(0) - (b >> np.uint64(shift))) & m
    if shift:   # lower bits are already 0 in both
        assert not (a & np.uint64((1 << shift) - 1)).any() and not (b & np.uint64((1 << shift) - 1)).any()
    order = np.argsort(kb, kind="stable")
    lo = np.searchsorted(kb[order], ka, "left")
    n = np.searchsorted(kb[order], ka, "right") - lo
    x = np.repeat(np.arange(a.size), n)
    y = order[np.repeat(lo, n) + np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n)]
    return a[x] + b[y], np.concatenate([ia[x], ib[y]], axis=1)


def _equal_sums(first, per):
    """Two sets of four ids >= first with equal sums of mix64 modulo 2^64, by
    Wagner's generalised birthday method on eight lists of `per` ids."""
    lists = []
    for i in range(8):
        ids = np.arange(first + i * per, first + (i + 1) * per, dtype=np.int64)
        v = _mix64(ids)
        lists.append((v if i < 4 else np.uint64(0) - v, ids[:, None]))
    for bits, shift in ((16, 0), (16, 16), (32, 32)):
        lists = [_join(lists[i][0], lists[i + 1][0], lists[i][1], lists[i + 1][1], bits, shift)
                 for i in range(0, len(lists), 2)]
    s, ids = lists[0]
    assert s.size and not s[0]
    return np.sort(ids[0, :4]), np.sort(ids[0, 4:])


def test_equal_content_keys():
    """Vertices 0 and 1 merge and no others can (each has an inbound pin and
    Phi is 1), so the next level's id of v >= 2 is v - 1: two hyperedges of
    one source whose destinations' hashes there have equal sums."""
    per = 80_000
    first = 3
    a, b = _equal_sums(first, per)
    assert _mix64(a).sum() == _mix64(b).sum() and not np.intersect1d(a, b).size
    V = first + 8 * per + 3
    x, y = V - 2, V - 1
    hg = _net("equalkeys", V, [(0, [1]), (x, a + 1), (x, b + 1), (x, [y]), (y, [x])], [7, 3, 5, 2, 1],
              64, 64, 1)
    assert lockstep(hg, max_levels=1) == 1


@pytest.mark.parametrize("starts", [1, 3, 40])
@pytest.mark.parametrize("n, hedges", [(21, 5400), (21, 1600), (64, 1500)])
def test_initial_placement_swaps(n, hedges, starts):
    """Swaps of nodes with at least 512 hyperedges a pair: a cluster per job
    while there are few jobs, a block with more (40 starts at the deeper
    levels) or with fewer hyperedges."""
    import paper_2609_07577_gb300 as P
    rng = np.random.default_rng(n + hedges)
    pins, off = [], [0]
    for _ in range(hedges):
        p = rng.choice(n, int(rng.integers(2, 5)), replace=False)
        pins.append(p)
        off.append(off[-1] + p.size)
    off, pins = np.asarray(off, np.int64), np.concatenate(pins).astype(np.int32)
    eta = rng.integers(1, 30, hedges).astype(np.int64)
    width = height = 8
    seq0 = np.stack([rng.permutation(n) for _ in range(starts)]).astype(np.int32)
    gamma = torch.empty((starts, n), dtype=torch.int32, device="cuda")
    P.snnmap_place_initial(n, hedges, torch.tensor(off).cuda(), torch.tensor(pins).cuda(),
                           torch.tensor(eta).cuda(), width, height, starts,
                           torch.tensor(seq0).cuda(), gamma)
    torch.cuda.synchronize()
    got = gamma.cpu().numpy()
    for s in range(starts):
        assert np.array_equal(got[s], oracle.initial_placement(n, off, pins, eta, width, height, seq0[s]))


def test_batch_of_uneven_partition_counts():
    """Jobs at once whose kernels keep different amounts of shared memory a
    block: each result equals the handle's own pass."""
    import dataclasses
    from paper_2609_07577_gb300 import HGraph, batch_partition
    hgs = []
    for name in ("cfg1", "cfg2s"):
        hg = snngen.by_name(name)
        for f in (1, 3, 8, 20, 40, 64):
            hgs.append(dataclasses.replace(hg, omega=hg.omega * f, delta=hg.delta * f, phi=hg.phi * f))
    rc, rs = batch_partition(hgs, slots=6)
    assert rc == 0, [r.get("error") for r in rs]
    for hg, r in zip(hgs, rs):
        G = HGraph.from_hypergraph(hg)
        rho, cost, _ = G.partition()
        G.close()
        assert r["cost"] == cost
        assert np.array_equal(np.asarray(r["rho"].cpu() if hasattr(r["rho"], "cpu") else r["rho"]),
                              rho.cpu().numpy())
