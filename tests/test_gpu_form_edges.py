"""More sizes at which the CUDA kernels change form (see test_gpu_edges.py):

- counters of incidence lists in shared memory up to 49,152 vertices, the
  histograms' plan in one launch up to 65,536;
- connection rows of more than 8,192 partitions (chunks of more than one step);
- the count pass over a round's hyperedges in one launch up to a bound of
  32,768 of them;
- the mark of a short prefix's hyperedges from the pin counts up to 2^24 pins.
"""
import numpy as np
import pytest
import torch

import oracle
import snngen
from gpu_helpers import lockstep
from test_gpu_edges import _lib, _net, _same_pass  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [49152, 49153, 65536, 65537])
def test_vertex_counts(V):
    rng = np.random.default_rng(V)
    src = rng.choice(V, 9000, replace=False)
    hedges = [(int(s), rng.choice(V, 6)) for s in src] + [(0, rng.choice(V, 1500)), (V - 1, np.arange(5))]
    hg = _net("vertices", V, hedges, rng.integers(1, 9, len(hedges)), 30, 500, 2000)
    assert lockstep(hg, max_levels=2) == 2


def test_rows_of_many_partitions():
    hg = snngen.layered(4, 5000, 8, 4, seed=3, omega=2, delta=64, phi=256, name="pairs")
    logs = _same_pass(hg)
    rho, _, st, _, _ = oracle.partition(hg, oracle.params_of(hg))
    assert st["n_parts"] > 8192 and any(r["rows"] for r in logs)


@pytest.mark.parametrize("E", [32767, 32768, 32769])
def test_recount_bound(E):
    """A first round that proposes moves of most vertices (the bound is then E)
    and later ones of few."""
    from paper_2609_07577_gb300 import HGraph, params_for
    rng = np.random.default_rng(E)
    V, K = 12000, 40
    hedges = [(int(a), rng.choice(V, 3)) for a in rng.integers(0, V, E)]
    hg = _net("recount", V, hedges, rng.integers(1, 9, E), 2 * V // K, 1 << 20, 1 << 20)
    prm = oracle.params_of(hg)
    want = (rng.permutation(V) % K).astype(np.int32)
    G = HGraph.from_hypergraph(hg, params=params_for(hg.omega, hg.delta, hg.phi))
    try:
        rho = torch.from_numpy(want.copy()).cuda()
        cost = G.refine(0, K, rho)
    finally:
        G.close()
    L = oracle.Level.from_hypergraph(hg, prm)
    rounds, moves, _ = L.refine(K, want, prm)
    assert rounds >= 2 and moves > 0
    assert np.array_equal(rho.cpu().numpy(), want) and cost == L.conn(want)


def test_prefix_marks():
    """2^24 pins exactly, and with two more in a hyperedge of weight 0 that no
    limit notices: the same moves by either form."""
    import paper_2609_07577_gb300 as P
    from paper_2609_07577_gb300 import HGraph, params_for
    rng = np.random.default_rng(7)
    V, E, K = 8192, 4096, 6
    step = 2 * rng.integers(0, V // 2, E) + 1   # odd: the pins of a hyperedge are distinct
    first = rng.integers(0, V, E)
    pins = ((first[:, None] + step[:, None] * np.arange(4096)) % V).astype(np.int32).ravel()
    off = np.arange(E + 1, dtype=np.int64) * 4096
    w = rng.integers(1, 100, E).astype(np.int32)
    small = 6000   # hyperedges of two pins decide the gains: the long ones reach every part
    a = rng.integers(0, V, small)
    b = (a + 1 + rng.integers(0, V - 1, small)) % V
    tail = np.stack([a, b], 1).astype(np.int32).ravel()
    pins = np.concatenate([pins[:(E - 3) * 4096], tail])   # 12,288 = 3 * 4096 pins, 12,000 used
    fill = (1 << 24) - pins.size
    pins = np.concatenate([pins, np.arange(fill, dtype=np.int32)])
    off = np.concatenate([off[:E - 2], off[E - 3] + 2 * np.arange(1, small + 1), [1 << 24]])
    w = np.concatenate([w[:E - 3], rng.integers(1, 9, small).astype(np.int32), [1]]).astype(np.int32)
    assert off[-1] == pins.size == 1 << 24 and off.size == w.size + 1
    start = torch.from_numpy((rng.permutation(V) % K).astype(np.int32)).cuda()

    def run(off, pins, w):
        dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (off, pins, w)]
        G = HGraph(params_for(2 * V // K, 1 << 28, 1 << 28), V, *dev)
        try:
            rho = start.clone()
            cost = G.refine(0, K, rho)
            assert P.snnmap_connectivity(G.handle, K, rho) == cost
            return rho, cost, [(r["istar"], r["gain"]) for r in G.round_logs()]
        finally:
            G.close()
    one = run(off, pins, w)
    two = run(np.append(off, off[-1] + 2), np.append(pins, np.array([0, 1], np.int32)),
              np.append(w, np.int32(0)))
    assert torch.equal(one[0], two[0]) and one[1:] == two[1:]
    assert len(one[2]) >= 2 and one[2][0][0] > 0
