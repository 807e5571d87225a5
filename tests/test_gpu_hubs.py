"""Placement of hypergraphs with nodes in many hyperedges, whose incidence
lists the kernels cut into pieces: degrees at the edges of a piece (512 for a
warp per node, 4,096 for a block per node) and of several, against the oracle
start by start (whole numbers: equal)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def hub_case(rng, n, degrees):
    """Node h is in exactly degrees[h] hyperedges, the others in what is left."""
    others = np.arange(len(degrees), n)
    hedges = []
    for h, d in enumerate(degrees):
        for _ in range(d):
            hedges.append(np.append(rng.choice(others, int(rng.integers(1, 3)), replace=False), h))
    for p in hedges:
        rng.shuffle(p)
    off = np.concatenate([[0], np.cumsum([len(p) for p in hedges])]).astype(np.int64)
    return off, np.concatenate(hedges).astype(np.int32), rng.integers(1, 30, len(hedges)).astype(np.int64)


@pytest.mark.parametrize("n, starts, degrees", [
    (76, 64, (511, 512, 513, 1024, 1025, 1536, 3000)),
    (24, 2, (4095, 4096, 4097)), (24, 3, (8192, 8193)), (24, 1, (13000,))])
def test_hubs(n, starts, degrees):
    import paper_2609_07577_gb300 as P
    rng = np.random.default_rng(n + starts)
    off, pins, eta = hub_case(rng, n, degrees)
    assert list(np.bincount(pins)[:len(degrees)]) == list(degrees)
    width = height = int(np.ceil(np.sqrt(n))) + 1
    dev = [torch.from_numpy(x).cuda() for x in (off, pins, eta)]
    seq0 = np.stack([rng.permutation(n) for _ in range(starts)]).astype(np.int32)
    gamma = torch.empty((starts, n), dtype=torch.int32, device="cuda")
    P.snnmap_place_initial(n, len(eta), *dev, width, height, starts, torch.from_numpy(seq0).cuda(), gamma)
    first = gamma.cpu().numpy().copy()
    rounds, logs = P.snnmap_place_refine(n, len(eta), *dev, width, height, starts, gamma, 1000, log_cap=4096)
    got = gamma.cpu().numpy()
    assert np.array_equal(first[-1], oracle.initial_placement(n, off, pins, eta, width, height, seq0[-1]))
    moved = 0
    for s in sorted({0, starts // 2, starts - 1}):
        want, want_logs = oracle.place_refine(n, off, pins, eta, width, height, first[s])
        assert np.array_equal(got[s], want)
        assert rounds[s] == len(want_logs) and logs[s] == want_logs
        moved += any(r["applied"] for r in want_logs)
    assert moved
