"""Performance cases: what users of the library have it do, through its public entry points.

Each case names a kind of call (``kind``) and its sizes.  The inputs are synthetic hypergraphs of the
benchmark's shapes (uniform with geometric edge sizes, VLSI-netlist-like with power-law sizes and locality,
row-nets with log-normal rows and hub rows, graphs of two-pin edges), made on the GPU from the seed alone.
All results are whole numbers and identical from run to run, so they are compared for equality.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2504_12013_gb300 import jet, synth

SCHEDULE = ((3, 4), (3, 8), (0, 1))  # the temperatures of Algorithm 1 (Section 7.2)
LIMIT = 8                            # iterations without improvement that end a temperature
TAU = (3, 4)                         # single iterations run at the first temperature
COARSEST_PER_BLOCK = 160             # coarsening weight bound: c(V) / (160 k)

# one row per shape: mean pins of an edge, for the byte counts of work()
GEO = {"geo12": (1, 2, 64), "geo25": (2, 5, 256)}  # |e| = 2 + Geometric(p) failures, capped
VLSI_MAX = 5000


def listed():
    return [
        # the plain small call: Algorithm 1 to convergence on 10,000 vertices; latency and launches count
        {"name": "refine_10k", "kind": "refine", "shape": "geo12", "n": 10_000, "m": 12_000, "k": 8, "c_max": 1,
         "w_max": 1},
        # a mid-sized call with every weight in use, odd sizes and a k that is no power of two
        {"name": "refine_100k_weighted", "kind": "refine", "shape": "geo25", "n": 100_003, "m": 110_017, "k": 37,
         "c_max": 8, "w_max": 4},
        # the largest one-GPU workload: eight Jet iterations on a row-net with hub rows
        {"name": "rounds_rownet_4m", "kind": "rounds", "shape": "rownet", "n": 4_000_000, "m": 4_000_000, "k": 128,
         "c_max": 1, "w_max": 1, "rounds": 8},
        # the VLSI-like workload: eight Jet iterations, vertex weights 1..4
        {"name": "rounds_vlsi_2m", "kind": "rounds", "shape": "vlsi", "n": 2_000_000, "m": 2_200_000, "k": 64,
         "c_max": 4, "w_max": 1, "rounds": 8},
        # many blocks (two 128-bit mask halves per edge), weighted edges, odd sizes
        {"name": "rounds_300k_k200", "kind": "rounds", "shape": "geo25", "n": 300_007, "m": 330_011, "k": 200,
         "c_max": 8, "w_max": 20, "rounds": 4},
        # plain graphs on the graph path (no pin counts): eight Jet iterations
        {"name": "graph_4m", "kind": "graph", "shape": "graph", "n": 4_000_000, "m": 16_000_000, "k": 64, "c_max": 1,
         "w_max": 1, "rounds": 8},
        # rebalancing alone: a partition whose low blocks have grown too heavy
        {"name": "rebalance_500k", "kind": "rebalance", "shape": "geo25", "n": 500_009, "m": 550_000, "k": 27,
         "c_max": 8, "w_max": 1},
        # many small instances refined by one persistent launch
        {"name": "batch_48", "kind": "batch", "shape": "geo25", "n": 60_000, "m": 66_000, "k": 32, "c_max": 1,
         "w_max": 1, "count": 48},
        # one served request: host buffers in, refined partition out, everything set up and freed inside
        {"name": "host_job_130k", "kind": "host", "shape": "geo25", "n": 129_871, "m": 142_858, "k": 32, "c_max": 8,
         "w_max": 1},
        # one coarsening level: clustering and contraction
        {"name": "coarsen_vlsi_500k", "kind": "coarsen", "shape": "vlsi", "n": 500_000, "m": 550_000, "k": 64,
         "c_max": 4, "w_max": 1},
        # what a finished partition is asked for: pin counts, (lambda-1), the matching schedule of its blocks
        {"name": "analyse_vlsi_1m", "kind": "analyse", "shape": "vlsi", "n": 1_000_000, "m": 1_100_000, "k": 128,
         "c_max": 4, "w_max": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("refine", "rounds", "rounds", "graph", "rebalance", "batch", "host", "coarsen",
                       "analyse"))
    shape = rng.choice(("geo12", "geo25", "vlsi"))
    k = _log(rng, 2, 256)
    c_max, w_max = rng.choice(((1, 1), (4, 1), (8, 4), (8, 20)))
    case = {"kind": kind, "shape": shape, "k": k, "c_max": c_max, "w_max": w_max}
    if kind == "refine":
        n = _log(rng, 1_000, 200_000)
    elif kind == "rounds":
        case["shape"] = rng.choice(("geo25", "vlsi", "rownet"))
        n = _log(rng, 10_000, 2_000_000)
        case["rounds"] = rng.choice((1, 2, 4, 8))
    elif kind == "graph":
        case["shape"] = "graph"
        n = _log(rng, 10_000, 4_000_000)
        case["rounds"] = rng.choice((1, 2, 4, 8))
    elif kind == "rebalance":
        n = _log(rng, 5_000, 1_000_000)
    elif kind == "batch":
        n = _log(rng, 4_000, 100_000)
        case.update(shape="geo25", c_max=1, w_max=1, k=rng.choice((2, 8, 32)), count=rng.randint(8, 48))
    elif kind == "host":
        n = _log(rng, 2_600, 500_000)
        case["shape"], case["k"] = "geo25", 2 << rng.randrange(8)
    elif kind == "coarsen":
        n = _log(rng, 10_000, 500_000)
    else:
        n = _log(rng, 10_000, 1_000_000)
    case["n"] = n
    case["m"] = n if case["shape"] == "rownet" else 4 * n if case["shape"] == "graph" else int(round(1.1 * n))
    return case


# ------------------------------------------------------------------ inputs

def _hubs(n):
    """Hub rows of a row-net of n rows: how many, and their range of lengths (200 of 50k..200k at 4M)."""
    return max(1, n // 20_000), max(2, n // 80), max(3, n // 20)


def _vlsi_table(n):
    s = np.arange(2, min(VLSI_MAX, max(2, n // 4)) + 1, dtype=np.float64)
    w = s ** -2.5
    return s, w / w.sum()


def _mean_pins(case):
    shape, n = case["shape"], case["n"]
    if shape in GEO:
        a, b, _ = GEO[shape]
        return 2 + (b - a) / a
    if shape == "vlsi":
        s, w = _vlsi_table(n)
        return float((s * w).sum())
    if shape == "rownet":
        count, lo, hi = _hubs(n)
        return math.exp(2.5) + count * (lo + hi) / 2 / case["m"]
    return 2.0


def _hypergraph(case, gen):
    """Both CSR views on the GPU; the pins of an edge are distinct and ascending."""
    n, m, shape = case["n"], case["m"], case["shape"]
    dev = gen.device
    rand = lambda size: torch.rand(size, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    whole = lambda hi, size: torch.randint(hi, (size,), generator=gen, device=dev)  # noqa: E731
    if shape == "graph":  # 80 % of the edges reach at most 1,000 ids away
        u = whole(n, m)
        far = torch.where(rand(m) < 0.8, 1 + whole(min(1000, n - 1), m), 1 + whole(n - 1, m))
        v = (u + far) % n
        pins = torch.stack((torch.minimum(u, v), torch.maximum(u, v)), dim=1).reshape(-1)
        sizes = torch.full((m,), 2, dtype=torch.int64, device=dev)
        eid = torch.arange(m, device=dev).repeat_interleave(2)
    else:
        if shape in GEO:
            a, b, cap = GEO[shape]
            sizes = 2 + torch.floor(torch.log1p(-rand(m)) / math.log(1 - a / b)).long()
            sizes = sizes.clamp(max=cap)
        elif shape == "vlsi":
            s, w = _vlsi_table(n)
            cdf = torch.from_numpy(np.cumsum(w)).to(dev)
            sizes = 2 + torch.searchsorted(cdf, rand(m)).clamp(max=len(s) - 1)
        else:
            normal = torch.randn(m, generator=gen, device=dev, dtype=torch.float64)
            sizes = torch.exp(2 + normal).round().long().clamp(1, n)
            count, lo, hi = _hubs(n)
            sizes[torch.randperm(m, generator=gen, device=dev)[:count]] = lo + whole(hi - lo, count)
        eid = torch.arange(m, device=dev).repeat_interleave(sizes)
        pins = whole(n, eid.numel())
        if shape == "vlsi":  # 80 % of the pins lie within 1 % of the ids around the edge's centre
            window = max(2, n // 100)
            near = (whole(n, m)[eid] + whole(2 * window + 1, eid.numel()) - window) % n
            pins = torch.where(rand(eid.numel()) < 0.8, near, pins)
        key = torch.unique(eid * n + pins)  # sorted: by edge, then pin, repeated pins dropped
        eid, pins = key // n, key % n
        sizes = torch.bincount(eid, minlength=m)
        del key
    zero = torch.zeros(1, dtype=torch.int64, device=dev)
    eptr = torch.cat((zero, torch.cumsum(sizes, 0)))
    vptr = torch.cat((zero, torch.cumsum(torch.bincount(pins, minlength=n), 0)))
    inc = (torch.sort(pins * m + eid).values % m).to(torch.int32)
    vwgt = (1 + whole(case["c_max"], n)).to(torch.int32)
    ewgt = (1 + whole(case["w_max"], m)).to(torch.int32)
    return jet.DeviceHypergraph.from_tensors(n, m, pins.numel(), eptr, pins.to(torch.int32), vptr, inc, vwgt, ewgt)


def _partition(n, k, gen):
    """A balanced random partition."""
    part = torch.empty(n, dtype=torch.int32, device=gen.device)
    part[torch.randperm(n, generator=gen, device=gen.device)] = \
        (torch.arange(n, device=gen.device) % k).to(torch.int32)
    return part


def _cmax(hg, k):
    """Weight bound of a coarsening level."""
    return max(1, min(32767, -(-int(hg.vwgt.sum()) // (COARSEST_PER_BLOCK * k))))


def _pinned(tensor):
    return tensor.cpu().pin_memory().numpy()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, k = case["kind"], case["k"]
    s = SimpleNamespace(kind=kind, case=case)
    if kind == "batch":  # instances of n/16 .. n vertices, evenly spread over the logarithm
        s.ctxs, parts = [], []
        for i in range(case["count"]):
            n = int(case["n"] / 16 ** (i / case["count"]))
            hg = _hypergraph(dict(case, n=n, m=int(round(n * case["m"] / case["n"]))), gen)
            s.ctxs.append(jet.jet_ctx_create(hg, jet.params(k)))
            parts.append(_partition(n, k, gen))
        # the states are slices, 256 bytes aligned, of one buffer each
        up = lambda x: -(-x // 64) * 64  # noqa: E731
        s.init = torch.cat([torch.nn.functional.pad(p, (0, up(p.numel()) - p.numel())) for p in parts])
        s.part = torch.empty_like(s.init)
        s.phi = torch.zeros(sum(up(c.hg.m * k) for c in s.ctxs), dtype=torch.int32, device="cuda")
        s.block_w = torch.zeros(len(s.ctxs), k, dtype=torch.int64, device="cuda")
        s.states, at, at_phi = [], 0, 0
        for i, c in enumerate(s.ctxs):
            s.states.append(SimpleNamespace(part=s.part[at:at + c.hg.n], phi=s.phi[at_phi:at_phi + c.hg.m * k],
                                            block_w=s.block_w[i]))
            at, at_phi = at + up(c.hg.n), at_phi + up(c.hg.m * k)
        s.batch = jet.jet_batch_create(s.ctxs)
        jet.jet_batch_set_team(s.batch, 8, 1024, 0)
        return s
    s.hg = _hypergraph(case, gen)
    if kind == "coarsen":
        s.order = torch.randperm(case["n"], generator=gen, device="cuda").to(torch.int32)
        s.cmax = _cmax(s.hg, k)
        # where the program keeps its levels: the coarse arrays go into buffers of the input's sizes
        zeros = lambda count, dtype: torch.zeros(count, dtype=dtype, device="cuda")  # noqa: E731
        pins = int(1.5 * case["m"] * _mean_pins(case)) + 20_000
        s.level = {"eptr": zeros(case["m"] + 1, torch.int64), "pins": zeros(pins, torch.int32),
                   "vptr": zeros(case["n"] + 1, torch.int64), "inc": zeros(pins, torch.int32),
                   "vwgt": zeros(case["n"], torch.int32), "ewgt": zeros(case["m"], torch.int32)}
        return s
    if kind == "host":
        h = s.hg
        s.host = synth.Hypergraph(n=h.n, m=h.m, eptr=_pinned(h.eptr), pins=_pinned(h.pins), vptr=_pinned(h.vptr),
                                  inc=_pinned(h.inc), vwgt=_pinned(h.vwgt), ewgt=_pinned(h.ewgt))
        s.init = _pinned(_partition(h.n, k, gen))
        s.part = _pinned(torch.zeros(h.n, dtype=torch.int32))
        s.params = jet.params(k)
        del s.hg
        return s
    s.ctx = jet.jet_ctx_create(s.hg, jet.params(k))
    s.init = _partition(case["n"], k, gen)
    if kind == "graph":
        jet.jet_set_graph_path(s.ctx, True)
    if kind == "rebalance":  # an eighth of the vertices drifts to the lower third of the blocks
        drift = torch.rand(case["n"], generator=gen, device="cuda") < 0.125
        low = torch.randint(max(1, k // 3), (case["n"],), generator=gen, device="cuda").to(torch.int32)
        s.init = torch.where(drift, low, s.init)
    s.state = jet.JetState(s.ctx, s.init.clone(), with_phi=kind != "graph")
    if kind == "analyse":  # a partition that has been refined
        for _ in range(8):
            s.state.round(TAU)
        s.objective = torch.zeros(1, dtype=torch.int64, device="cuda")
    return s


# ------------------------------------------------------------------ calls

def _numbers(results):
    """The summaries of a call's instances as one array."""
    return np.array([[r["iterations"], r["objective"], r["initial_objective"], r["balanced"],
                      *r["phase_iterations"]] for r in results], dtype=np.int64)


def run(s):
    kind, case = s.kind, s.case
    if kind == "batch":
        s.part.copy_(s.init)
        res = jet.jet_batch_refine(s.batch, SCHEDULE, LIMIT, s.states)
        return {"part": s.part, "phi": s.phi, "block_w": s.block_w, "results": _numbers(res)}
    if kind == "host":
        s.part[:] = s.init
        res = jet.jet_refine_host(s.host, s.params, SCHEDULE, LIMIT, s.part)
        return {"part": s.part, "results": _numbers([res])}
    if kind == "coarsen":
        coarse, to_coarse, label = jet.jet_coarsen(s.hg, s.cmax, s.order)
        for name, kept in s.level.items():
            array = getattr(coarse, name)
            kept[:array.numel()].copy_(array)
        return dict(s.level, label=label, map=to_coarse, n=coarse.n, m=coarse.m, P=coarse.P)
    t = s.state
    if kind == "refine":
        t.part.copy_(s.init)
        res = jet.jet_refine(s.ctx, SCHEDULE, LIMIT, t.part, t.phi, t.block_w)
        return {"part": t.part, "phi": t.phi, "block_w": t.block_w, "results": _numbers([res])}
    if kind == "analyse":
        jet.jet_build_pincounts(s.ctx, t.part, t.phi, t.block_w)
        jet.jet_connectivity(s.ctx, t.phi, s.objective)
        pairs, round_of, rounds = jet.jet_quotient_schedule(s.ctx, t.phi)
        scheduled = np.zeros((3, s.ctx.k * (s.ctx.k - 1) // 2), dtype=np.int32)
        scheduled[:2, :len(pairs)], scheduled[2, :len(pairs)] = pairs.T, round_of
        return {"phi": t.phi, "block_w": t.block_w, "objective": s.objective, "scheduled": scheduled,
                "pairs": len(pairs), "rounds": rounds}
    t.part.copy_(s.init)
    jet.jet_build_pincounts(s.ctx, t.part, t.phi, t.block_w)
    if kind == "rebalance":
        jet.jet_rebalance(s.ctx, t.part, t.phi, t.block_w, t.stats)
        return {"part": t.part, "phi": t.phi, "block_w": t.block_w, "stats": t.stats}
    t.locked.zero_()
    for _ in range(case["rounds"]):
        t.round(TAU)
    out = {"part": t.part, "block_w": t.block_w, "locked": t.locked, "stats": t.stats}
    if t.phi is not None:
        out["phi"] = t.phi
    return out


def work(case):
    """The hypergraph and the partition read once, every output written once."""
    n, m, k, kind = case["n"], case["m"], case["k"], case["kind"]
    P = m * _mean_pins(case)
    graph = 8 * P + 12.0 * (n + m)
    if kind == "coarsen":
        return {"bytes": graph + 4 * n + 8 * n + graph / 4, "flops": 0}
    state = 8 * n + 8 * k + (0 if kind in ("graph", "host") else 4.0 * m * k)
    if kind == "batch":  # the mean size is n (1 - 1/16) / ln 16
        return {"bytes": case["count"] * (graph + state) * (15 / 16) / math.log(16), "flops": 0}
    if kind == "analyse":  # no partition is written; (lambda-1) reads the pin counts
        return {"bytes": 4 * P + 12.0 * (n + m) + state + 4.0 * m * k, "flops": 0}
    return {"bytes": graph + state, "flops": 0}


def exact(case, seed):
    """Every output is a whole number, compared for equality."""
    return None
