"""The work that users of this library have it do, as measurable cases.

Kinds of case (the size grows with the number of neurons; every kind goes
through the package's public entry points):

* ``pass``    one mapping job: build the handle from the network's arrays on
              the device, run the whole multilevel pass, give the handle back.
              What ``python -m paper_2609_07577_gb300 map``, the benchmark and
              every request of the batched and served forms do.
* ``coarsen`` one ``coarsen_level`` of a kept level-0 handle (neighbour
              histograms, candidates, matching): the call of a program that
              drives the levels itself.
* ``refine``  ``refine`` of a partition in hand (the neurons in their natural
              order, in equal cores) on a kept handle: improving an existing
              mapping.
* ``graph``   the partition hypergraph of a partition in hand on a kept
              handle: what a placement starts from.
* ``place``   the multi-start placement of a partition hypergraph on its
              lattice of cores.
* ``batch``   several independent jobs of uneven sizes at once, on the
              batched form's slots.

The networks are the repository's three families (snngen): ``layered``
(window plus random picks), ``conv`` (3 x 3 receptive fields plus random
picks) and ``powerlaw`` (recurrent, heavy-tailed fan-out), drawn on the GPU.
Every output is a whole number.
"""
import math

import numpy as np
import torch

import paper_2609_07577_gb300 as snnmap

DEV = "cuda"
PLACE_STARTS = 64      # starts of a placement (the paper's and place()'s number)
BATCH_SLOTS = 8        # batch_partition's own default


def listed():
    return [
        # the smallest network in use: latency and launches
        {"name": "pass_layered_4k", "kind": "pass", "net": "layered", "width": 1024, "omega": 256,
         "delta": 64, "phi": 4096},
        # a small recurrent network (the served form's lower end)
        {"name": "pass_powerlaw_10k", "kind": "pass", "net": "powerlaw", "V": 10007,
         "block": 4096, "fmax": 2048, "omega": 512, "delta": 2048, "phi": 8192},
        # an ordinary feedforward job of the batched workload, at an odd width
        {"name": "pass_layered_60k", "kind": "pass", "net": "layered", "width": 15013,
         "omega": 1024, "delta": 4096, "phi": 16384},
        # an ordinary conv job
        {"name": "pass_conv_66k", "kind": "pass", "net": "conv", "layers": 8, "side": 32,
         "omega": 1024, "delta": 4096, "phi": 16384},
        # an ordinary recurrent job with large cores (the slowest kind per neuron)
        {"name": "pass_powerlaw_12k", "kind": "pass", "net": "powerlaw", "V": 12007,
         "block": 65536, "fmax": 16384, "omega": 4096, "delta": 16384, "phi": 65536},
        # the benchmark's network: the largest whole pass
        {"name": "pass_conv_1m", "kind": "pass", "net": "conv", "layers": 8, "side": 128,
         "omega": 1024, "delta": 4096, "phi": 16384},
        # the histogram of the benchmark's network, one call
        {"name": "coarsen_conv_1m", "kind": "coarsen", "net": "conv", "layers": 8, "side": 128,
         "omega": 1024, "delta": 4096, "phi": 16384},
        # the histogram under skewed degrees
        {"name": "coarsen_powerlaw_1m", "kind": "coarsen", "net": "powerlaw", "V": 1 << 20,
         "block": 65536, "fmax": 16384, "omega": 4096, "delta": 16384, "phi": 65536},
        # an existing mapping improved
        {"name": "refine_conv_262k", "kind": "refine", "net": "conv", "layers": 8, "side": 64,
         "omega": 1024, "delta": 4096, "phi": 16384, "core": 128},
        # the partition hypergraph of the benchmark's network
        {"name": "graph_conv_1m", "kind": "graph", "net": "conv", "layers": 8, "side": 128,
         "omega": 1024, "delta": 4096, "phi": 16384, "core": 512},
        # a placement of ordinary size (the paper's networks end as 16 to
        # 1.7 thousand partitions)
        {"name": "place_256", "kind": "place", "net": "conv", "layers": 8, "side": 32,
         "omega": 1024, "delta": 4096, "phi": 16384, "core": 256},
        # the batched form: uneven sizes, both families
        {"name": "batch_4", "kind": "batch", "jobs": 4, "nmin": 10000, "nmax": 15000},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_conv(rng, kind, lo, hi):
    """A conv network of about lo to hi neurons (side from the size)."""
    layers = rng.choice([4, 6, 8])
    side = max(8, int(round(math.sqrt(_log_uniform(rng, lo, hi) / (8.0 * layers)))))
    return {"kind": kind, "net": "conv", "layers": layers, "side": side, "omega": 1024,
            "delta": 4096, "phi": 16384}


def draw(rng):
    k = rng.choice(["pass_layered", "pass_conv", "pass_powerlaw", "coarsen_conv",
                    "coarsen_powerlaw", "refine", "graph", "place", "batch"])
    if k == "pass_layered":
        omega = rng.choice([256, 1024, 4096])
        top = 12000 if omega < 4096 else 4000
        return {"kind": "pass", "net": "layered", "width": _log_uniform(rng, 1024, top),
                "omega": omega, "delta": 4 * omega, "phi": 16 * omega}
    if k == "pass_conv":
        return _draw_conv(rng, "pass", 8000, 400000)
    if k == "pass_powerlaw":
        omega = rng.choice([512, 1024, 4096])
        V = _log_uniform(rng, 5000, 12000 if omega < 4096 else 6000)
        return {"kind": "pass", "net": "powerlaw", "V": V, "block": rng.choice([4096, 65536]),
                "fmax": rng.choice([2048, 16384]), "omega": omega, "delta": 4 * omega,
                "phi": 16 * omega}
    if k == "coarsen_conv":
        return _draw_conv(rng, "coarsen", 8000, 1000000)
    if k == "coarsen_powerlaw":
        return {"kind": "coarsen", "net": "powerlaw", "V": _log_uniform(rng, 10000, 1 << 20),
                "block": rng.choice([4096, 65536]), "fmax": 16384, "omega": 4096,
                "delta": 16384, "phi": 65536}
    if k == "refine":
        return dict(_draw_conv(rng, "refine", 8000, 262144), core=rng.choice([96, 128]))
    if k == "graph":
        return dict(_draw_conv(rng, "graph", 8000, 1000000), core=rng.choice([128, 256, 512]))
    if k == "place":
        return dict(_draw_conv(rng, "place", 8000, 65536), core=rng.choice([256, 512]))
    nmin = _log_uniform(rng, 5000, 10000)
    return {"kind": "batch", "jobs": rng.randint(2, 4), "nmin": nmin, "nmax": int(1.5 * nmin)}


# ---------------------------------------------------------------------------
# networks, drawn on the GPU: (V, off int64[E+1], pins int32[P], w int32[E]),
# pin 0 of a hyperedge its source, then its distinct destinations ascending

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _assemble(V, src, hid, dst, w):
    """CSR from (hyperedge, destination) pairs in any order; repeated pairs
    and a source among its own destinations count once and not at all."""
    E = src.numel()
    key = torch.unique(hid[dst != src[hid]] * V + dst[dst != src[hid]])
    h, d = key // V, key % V
    cnt = torch.bincount(h, minlength=E) + 1
    off = torch.zeros(E + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(cnt, 0)
    pins = torch.empty(E + h.numel(), dtype=torch.int32, device=DEV)
    pins[off[:-1]] = src.to(torch.int32)
    # the j-th pair overall follows h + 1 sources
    pins[torch.arange(h.numel(), device=DEV) + h + 1] = d.to(torch.int32)
    return V, off, pins, w.to(torch.int32)


def _layered(c, seed, layers=4, window=32, nrand=8):
    g = _generator(seed)
    width = c["width"]
    E = (layers - 1) * width
    src = torch.arange(E, device=DEV)
    nxt = (src // width + 1) * width
    win = nxt[:, None] + (src[:, None] % width + torch.arange(window, device=DEV)) % width
    rnd = nxt[:, None] + torch.randint(0, width, (E, nrand), generator=g, device=DEV)
    w = torch.poisson(torch.full((E,), 5.0, device=DEV), generator=g) + 1
    dst = torch.cat([win, rnd], 1)
    return _assemble(layers * width, src, src[:, None].expand_as(dst).reshape(-1), dst.reshape(-1), w)


def _conv(c, seed, channels=8, nrand=4):
    g = _generator(seed)
    side, layers = c["side"], c["layers"]
    S = side * side * channels
    E = (layers - 1) * S
    src = torch.arange(E, device=DEV)
    nxt = (src // S + 1) * S
    cell = src % S // channels
    d = torch.tensor([-1, 0, 1], device=DEV)
    yy = (cell // side)[:, None] + d.repeat_interleave(3)
    xx = (cell % side)[:, None] + d.repeat(3)
    base = nxt[:, None] + (yy % side * side + xx % side) * channels
    win = (base[..., None] + torch.arange(channels, device=DEV)).reshape(E, -1)
    rnd = nxt[:, None] + torch.randint(0, S, (E, nrand), generator=g, device=DEV)
    u = torch.rand(E, generator=g, device=DEV, dtype=torch.float64)
    w = torch.floor(torch.log1p(-u) / math.log(0.8)) + 1     # geometric, p = 0.2
    dst = torch.cat([win, rnd], 1)
    return _assemble(layers * S, src, src[:, None].expand_as(dst).reshape(-1), dst.reshape(-1), w)


def _powerlaw(c, seed, fmin=8, alpha=2.1, local=0.7):
    g = _generator(seed)
    V, block = c["V"], min(c["block"], c["V"])
    f64 = torch.float64
    u = torch.rand(V, generator=g, device=DEV, dtype=f64)
    lo, hi = float(fmin) ** -alpha, float(c["fmax"]) ** -alpha
    fan = torch.floor((lo - u * (lo - hi)) ** (-1.0 / alpha)).to(torch.int64).clamp(fmin, c["fmax"])
    src = torch.arange(V, device=DEV)
    hid = torch.repeat_interleave(src, fan)
    n = hid.numel()
    is_local = torch.rand(n, generator=g, device=DEV) < local
    start = hid // block * block
    wide = torch.clamp(V - start, max=block)
    loc = start + torch.randint(0, block, (n,), generator=g, device=DEV) * wide // block
    uni = torch.randint(0, V, (n,), generator=g, device=DEV)
    z = torch.randn(V, generator=g, device=DEV, dtype=f64)
    w = torch.exp(1.0 + z).round().clamp(1, 2 ** 30)
    return _assemble(V, src, hid, torch.where(is_local, loc, uni), w)


def _network(c, seed):
    return {"layered": _layered, "conv": _conv, "powerlaw": _powerlaw}[c["net"]](c, seed)


def _params(c):
    return snnmap.params_for(c["omega"], c["delta"], c["phi"])


class _Arrays:
    """A network's host arrays and limits, as JobBuffers takes them."""

    def __init__(self, net, c):
        self.V = net[0]
        self.off, self.pins, self.w = (t.cpu().numpy() for t in net[1:])
        self.omega, self.delta, self.phi = c["omega"], c["delta"], c["phi"]


def _batch_cases(c):
    """The jobs of a batch: sizes spread over [nmin, nmax] (their logarithm),
    layered and recurrent networks in turn, two core sizes."""
    out = []
    for j in range(c["jobs"]):
        t = j / max(1, c["jobs"] - 1)
        n = int(round(c["nmin"] * (c["nmax"] / c["nmin"]) ** t))
        omega = (256, 1024)[j // 2 % 2]
        lim = {"omega": omega, "delta": 4 * omega, "phi": 16 * omega}
        if j % 2 == 0:
            out.append(dict(lim, net="layered", width=n // 4))
        else:
            out.append(dict(lim, net="powerlaw", V=n, block=65536, fmax=16384))
    return out


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        bufs = []
        for j, jc in enumerate(_batch_cases(c)):
            bufs.append(snnmap.JobBuffers(_Arrays(_network(jc, 1000 * seed + j), jc),
                                          on_host=False))
        return {"case": c, "bufs": bufs}
    V, off, pins, w = _network(c, seed)
    if c["kind"] == "pass":
        return {"case": c, "params": _params(c), "V": V, "off": off, "pins": pins, "w": w}
    G = snnmap.HGraph(_params(c), V, off, pins, w)
    if c["kind"] == "coarsen":
        i32, i64 = torch.int32, torch.int64
        out = [torch.empty(V, dtype=t, device=DEV) for t in (i32, i64, i32, i32)]
        return {"case": c, "G": G, "out": out}
    rho = (torch.arange(V, device=DEV) // c["core"]).to(torch.int32)
    parts = -(-V // c["core"])
    if c["kind"] == "place":
        gp = G.partition_graph(rho, parts)
        G.close()
        return {"case": c, "parts": parts, "seed": seed,
                **{k: torch.from_numpy(gp[k]).to(DEV) for k in ("off", "pins", "eta")}}
    out = None
    if c["kind"] == "graph":
        # buffers that hold any partition hypergraph of such a network
        E = off.numel() - 1
        P = 77 * E   # a hyperedge has at most its source, 72 window and 4 random pins
        out = [torch.zeros(n, dtype=t, device=DEV)
               for n, t in ((E + 1, torch.int64), (P, torch.int32), (E, torch.int64),
                            (E, torch.int32))]
    return {"case": c, "G": G, "rho": rho, "parts": parts, "out": out}


def run(state):
    kind = state["case"]["kind"]
    if kind == "pass":
        G = snnmap.HGraph(state["params"], state["V"], state["off"], state["pins"], state["w"])
        rho, cost, stats = G.partition()
        G.close()
        return {"rho": rho, "cost": cost, "stats": stats}
    if kind == "coarsen":
        n_cand, n_pairs = state["G"].coarsen_level()
        snnmap.snnmap_last_matching(state["G"].handle, *state["out"])
        return {"n_cand": n_cand, "n_pairs": n_pairs, "out": state["out"]}
    if kind == "refine":
        rho = state["rho"].clone()
        return {"cost": state["G"].refine(0, state["parts"], rho), "rho": rho}
    if kind == "graph":
        h = state["G"].handle
        sizes = snnmap.snnmap_partition_graph(h, state["parts"], state["rho"])
        snnmap.snnmap_partition_graph_copy(h, *state["out"])
        return {"sizes": sizes, "out": state["out"]}
    if kind == "place":
        r = snnmap.place(state["parts"], state["off"], state["pins"], state["eta"],
                         n_starts=PLACE_STARTS, seed=state["seed"])
        return {k: np.asarray(r[k], dtype=np.int64)
                for k in ("gamma", "trd", "start", "rounds", "trds", "trds_initial")}
    rc, res = snnmap.batch_partition(None, slots=BATCH_SLOTS, buffers=state["bufs"])
    return {"rc": rc, "rho": [r["rho"] for r in res], "cost": [r["cost"] for r in res]}


# ---------------------------------------------------------------------------

def _sizes(c):
    """Expected (V, E, P, sum of |e|(|e| - 1)) of a network."""
    if c["net"] == "layered":
        width = c["width"]
        E, n = 3 * width, 33 + 8 * (1 - 36 / width)
        return 4 * width, E, E * n, E * n * (n - 1)
    if c["net"] == "conv":
        S = 8 * c["side"] ** 2
        E, n = (c["layers"] - 1) * S, 73 + 4 * (1 - 74 / S)
        return c["layers"] * S, E, E * n, E * n * (n - 1)
    # truncated Pareto fan-out x (first and second moment)
    V, a, m, M = c["V"], 2.1, 8.0, float(c["fmax"])
    k = a / (m ** -a - M ** -a)
    m1 = k * (m ** (1 - a) - M ** (1 - a)) / (a - 1) - 0.5
    m2 = k * (m ** (2 - a) - M ** (2 - a)) / (a - 2)
    return V, V, V * (m1 + 1), V * (m2 + m1)


def work(case):
    """Bytes: each input array read once and each output written once. flops:
    the integer additions no form of the path can do without (level 0's
    neighbour scores, one per pair of pins of a hyperedge; one count per pin
    for a partition's connections; one distance per pin pair of the
    partition hypergraph and start)."""
    c = case
    if c["kind"] == "batch":
        ws = [work(dict(j, kind="pass")) for j in _batch_cases(c)]
        return {k: sum(x[k] for x in ws) for k in ("bytes", "flops")}
    V, E, P, pairs = _sizes(c)
    net = 8 * (E + 1) + 4 * P + 4 * E
    if c["kind"] == "pass":
        return {"bytes": net + 4 * V, "flops": pairs}
    if c["kind"] == "coarsen":
        return {"bytes": net + 20 * V, "flops": pairs}
    if c["kind"] == "refine":
        return {"bytes": net + 8 * V, "flops": P}
    # an axon of a block of `core` neurons reaches about this many parts
    reach = min(V / c["core"], 6 * 32 / c["core"] ** 0.5 + 4)
    if c["kind"] == "graph":
        return {"bytes": net + 4 * V + E * (16 + 4 * reach), "flops": P}
    return {"bytes": E * (16 + 4 * reach) + 4 * PLACE_STARTS * V / c["core"],
            "flops": PLACE_STARTS * E * reach * reach}


def exact(case, seed):
    """Every output is a whole number (ids, counts, sums of whole weights):
    there is no rounding for a 64-bit evaluation to measure."""
    return None
