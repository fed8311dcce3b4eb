"""Measured calls of the engine: what a program that uses it has it do.

A case is a dict of plain values; ``prepare`` builds what such a program keeps
(handles, batches, result buffers), ``run`` makes one pass through the public
entry points, ``work`` counts what the pass cannot do without and ``exact``
restates the method in plain torch integers.  Four kinds of call:

  lattice   one lattice advanced by n sweeps, its E/M records and spins read
  batch     many lattices of mixed sizes in one persistent launch
  medium    one porous medium: porosity field, invasion, the cluster read
  media     many small media in one launch (spanning statistics)
"""
from __future__ import annotations

import math
from decimal import ROUND_FLOOR, Decimal, localcontext

import numpy as np
import torch

import paper_cs_0312006_gb300 as ising
from paper_cs_0312006_gb300 import batched, percolation, workloads

LAYOUTS = {"int8": ising.INT8, "packed": ising.BITPACK}
RULES = {"metropolis": ising.RULE_METROPOLIS, "heatbath": ising.RULE_HEATBATH,
         "multihit": ising.RULE_MULTIHIT, "demon": ising.RULE_DEMON}
STARTS = {"hot": ising.HOT, "cold": ising.COLD_UP}
QMAX = 3                 # demon capacity that both layouts take
DEMON_BETA = 0.5         # temperature of the initial demons
MAX_UPDATES = 1.34e9     # site updates of the largest listed lattice call


def lattice(name, dims, L, layout, sweeps, every, beta, rule="metropolis", start="hot", hits=1):
    case = {"kind": "lattice", "dims": dims, "L": L, "layout": layout, "rule": rule,
            "hits": hits, "beta": beta, "start": start, "sweeps": sweeps, "every": every}
    return {"name": name, **case} if name else case


def listed():
    b2, b3 = workloads.BETA_C_2D, workloads.BETA_C_3D
    return [
        # the smallest lattice of the paper's timings: a short critical run whose
        # cost is latency, E/M after every sweep
        lattice("square64_int8", 2, 64, "int8", 100, 1, b2),
        # a mid-sized square of the paper's timings in the layout the engine picks
        lattice("square512_packed", 2, 512, "packed", 50, 1, 0.44),
        # the large square of the temperature scan, cold start, both layouts
        lattice("square8192_int8", 2, 8192, "int8", 20, 1, 0.44, start="cold"),
        lattice("square8192_packed", 2, 8192, "packed", 20, 1, 0.44, start="cold"),
        # the critical cube, int8, E/M every tenth sweep
        lattice("cube256_int8", 3, 256, "int8", 20, 10, b3),
        # a ragged cube: rows that are neither whole words nor whole draw groups
        lattice("cube202_packed", 3, 202, "packed", 20, 10, 0.23),
        # the heat-bath rule on a ragged square of bytes
        lattice("square1000_heatbath_int8", 2, 1000, "int8", 50, 10, 0.42, rule="heatbath"),
        # several trials per visit
        lattice("square2048_multihit_packed", 2, 2048, "packed", 10, 1, 0.40, rule="multihit",
                hits=3),
        # the deterministic dynamics without draws
        lattice("square8192_demon_packed", 2, 8192, "packed", 20, 1, 0.44, rule="demon"),
        # independent lattices of mixed sizes, dimensions and temperatures
        {"name": "batch256", "kind": "batch", "lattices": 256, "mix": 0, "sweeps": 50},
        # one large medium just above the threshold: fluid from one face
        {"name": "medium4096", "kind": "medium", "dims": 2, "L": 4096, "porosity": 0.6,
         "source": "face"},
        # spanning statistics at the threshold
        {"name": "media256x2048", "kind": "media", "dims": 2, "L": 256, "porosity": 0.592746,
         "source": "face", "media": 2048},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(["lattice", "batch", "medium", "media"], [8, 1, 1, 2])[0]
    if kind == "lattice":
        dims = rng.choice([2, 2, 3])
        L = round(_log(rng, 16, 8192) if dims == 2 else _log(rng, 8, 320))
        if rng.random() < 0.4:  # many programs take whole powers or multiples of 32
            L = max(32, L // 32 * 32)
        L += L & 1
        rule = rng.choice(["metropolis"] * 4 + ["heatbath"] * 2 + ["multihit", "demon"])
        hits = rng.randint(2, 4) if rule == "multihit" else 1
        most = min(200, MAX_UPDATES / hits / L ** dims)
        every = 10 if most >= 10 and rng.random() < 0.5 else 1
        sweeps = max(1, int(_log(rng, max(1, every), max(every, most, 1)) / every)) * every
        centre = workloads.BETA_C_2D if dims == 2 else workloads.BETA_C_3D
        return lattice(None, dims, L, rng.choice(["int8", "packed"]), sweeps, every,
                       round(centre * rng.uniform(0.7, 1.3), 6), rule=rule,
                       start=rng.choice(["hot", "cold"]) if rule != "demon" else "hot", hits=hits)
    if kind == "batch":
        n = int(_log(rng, 8, 256))
        return {"kind": "batch", "lattices": n, "mix": rng.randrange(1000),
                "sweeps": 10 * rng.randint(1, 3)}
    if kind == "medium":
        dims = rng.choice([2, 3])
        threshold = 0.592746 if dims == 2 else 0.3116
        return {"kind": "medium", "dims": dims,
                "L": round(_log(rng, 100, 3000) if dims == 2 else _log(rng, 20, 200)),
                "porosity": round(threshold * rng.uniform(1.01, 1.3), 6),
                "source": rng.choice(["face", "point"])}
    dims = rng.choice([2, 2, 3])
    L = round(_log(rng, 16, 256) if dims == 2 else _log(rng, 8, 40))
    threshold = 0.592746 if dims == 2 else 0.3116
    most = min(2048, 2048 * 256 ** 2 / L ** dims)
    return {"kind": "media", "dims": dims, "L": L,
            "porosity": round(threshold * rng.uniform(0.98, 1.05), 6),
            "source": rng.choice(["face", "point"]), "media": max(1, int(_log(rng, 64, most)))}


def _engine_seed(seed):
    return workloads.BASE_SEED + 1_000_003 * seed


def _demons(n, seed):
    """Demons of 0..QMAX at DEMON_BETA, uint8, drawn through a table of 2^16."""
    w = np.exp(-4.0 * DEMON_BETA * np.arange(QMAX + 1))
    table = np.searchsorted(np.cumsum(w / w.sum())[:-1], (np.arange(65536) + 0.5) / 65536)
    draws = np.random.default_rng(seed).integers(0, 65536, n, dtype=np.uint16)
    return table.astype(np.uint8)[draws]


def _mix(case, seed):
    """The batch's lattices: shapes and temperatures from the case, draws from the seed."""
    specs = workloads.batched_mix(case["lattices"], case["sweeps"], case["mix"])
    for j, sp in enumerate(specs):
        sp.seed = _engine_seed(seed) + j
    return specs


def _site(case):
    """The invasion point: the middle of the medium."""
    L, dims = case["L"], case["dims"]
    return sum((L // 2) * L ** k for k in range(dims))


def _media_seeds(case, seed):
    return np.uint64(_engine_seed(seed)) + np.arange(case["media"], dtype=np.uint64)


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "lattice":
        n = case["L"] ** case["dims"]
        lat = ising.Lattice(case["dims"], case["L"], case["beta"], _engine_seed(seed),
                            layout=LAYOUTS[case["layout"]], start=STARTS[case["start"]])
        if case["rule"] == "multihit":
            lat.set_hits(case["hits"])
        if case["rule"] == "demon":
            lat.set_demons(_demons(n, seed), qmax=QMAX)
        lat.set_rule(RULES[case["rule"]])
        records = max(1, case["sweeps"] // case["every"])
        state.update(lat=lat, spins=torch.empty(n, dtype=torch.int8, device="cuda"),
                     pairs=torch.zeros((records, 2), dtype=torch.int64).pin_memory().numpy())
    elif kind == "batch":
        specs = _mix(case, seed)
        lats = batched.make_lattices(specs)
        at = np.cumsum([0] + [-(-sp.sites // 16) * 16 for sp in specs])
        records = sum(sp.sweeps // sp.measure_every for sp in specs)
        state.update(lats=lats, at=at.tolist(),
                     batch=ising.Batch(lats, [sp.sweeps for sp in specs],
                                       [sp.measure_every for sp in specs]),
                     spins=torch.zeros(int(at[-1]), dtype=torch.int8, device="cuda"),
                     pairs=torch.zeros((records, 2), dtype=torch.int64).pin_memory().numpy())
    elif kind == "medium":
        state.update(medium=percolation.Medium(case["dims"], case["L"], _engine_seed(seed)))
    else:
        n = case["media"] * case["L"] ** case["dims"]
        state.update(seeds=_media_seeds(case, seed),
                     clusters=torch.empty(n, dtype=torch.uint8, device="cuda"))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = state["lat"]
        lat.sweep(case["sweeps"], case["every"])
        n = lat.observables_async(state["pairs"])
        lat.get_spins_async(state["spins"].data_ptr())
        return {"records": state["pairs"][:n], "spins": state["spins"]}
    if kind == "batch":
        state["batch"].launch()
        state["batch"].sync()
        ising.observables_gather(state["lats"], state["pairs"])
        base = state["spins"].data_ptr()
        for lat, at in zip(state["lats"], state["at"]):
            lat.get_spins_async(base + at)
        return {"records": state["pairs"], "spins": state["spins"]}
    source = percolation.FACE if case["source"] == "face" else percolation.POINT
    if kind == "medium":
        medium = state["medium"]
        medium.generate(case["porosity"])
        r = medium.invade(source, _site(case))
        return {"size": r.size, "spans": r.spans, "steps": r.steps, "cluster": medium.cluster()}
    res = percolation.batch(case["dims"], case["L"], case["porosity"], state["seeds"], source,
                            _site(case), clusters_ptr=state["clusters"].data_ptr())
    return {"results": np.array([(r.size, r.spans, r.steps) for r in res], dtype=np.int64),
            "clusters": state["clusters"]}


def work(case):
    """Bytes: each colour pass reads its own and the other colour and writes its
    own; a medium's pores and cluster are written once.  Flops: integer
    operations of the draws, ten rounds of two multiplies and two xors for four
    sites (the demons' bit logic where nothing is drawn)."""
    kind = case["kind"]
    if kind == "lattice":
        updates = case["sweeps"] * case["L"] ** case["dims"]
        bits = 24 if case["layout"] == "int8" else 3
        if case["rule"] == "demon":
            bits = 40 if case["layout"] == "int8" else 7
        ops = 2 if case["rule"] == "demon" else 10 * case["hits"]
        return {"bytes": updates * bits / 8, "flops": updates * ops}
    if kind == "batch":
        updates = batched.total_updates(_mix(case, 0))
        return {"bytes": updates * 3 / 8, "flops": updates * 10}
    sites = case["L"] ** case["dims"] * case.get("media", 1)
    return {"bytes": sites * (1 / 8 + 1), "flops": sites * 10}


# ---- the method in plain torch integers ------------------------------------

MASK = 0xFFFFFFFF


def _mul(a, m):
    """High and low halves of the 64-bit products of 32-bit values by m."""
    ah = (a >> 16) * m
    low = ((ah & 0xFFFF) << 16) + (a & 0xFFFF) * m
    return (ah >> 16) + (low >> 32), low & MASK


def _draws(n, c1, c2, c3, seed):
    """The first n draws of the stream: word i & 3 of Philox4x32-10 at i >> 2."""
    c0 = torch.arange(-(-n // 4), dtype=torch.int64, device="cuda")
    c1, c2, c3 = (torch.full_like(c0, c) for c in (c1, c2, c3))
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        ahi, alo = _mul(c0, 0xD2511F53)
        bhi, blo = _mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = bhi ^ c1 ^ k0, blo, ahi ^ c3 ^ k1, alo
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return torch.stack([c0, c1, c2, c3], dim=1).reshape(-1)[:n]


def _thresholds(case):
    """Integer threshold by the number d of disagreeing neighbours."""
    dims, beta = case["dims"], Decimal(case["beta"])
    out = []
    with localcontext() as ctx:
        ctx.prec = 60
        for d in range(2 * dims + 1):
            e = (4 * beta * (dims - d)).exp()
            p = 1 / (1 + e) if case["rule"] == "heatbath" else min(Decimal(1), 1 / e)
            out.append(int((p * 2 ** 32).to_integral_value(ROUND_FLOOR)))
    return torch.tensor(out, dtype=torch.int64, device="cuda")


def _exact_lattice(case, seed):
    dims, L, rule = case["dims"], case["L"], case["rule"]
    W, rows, n, key = L // 2, L ** (dims - 1), L ** dims, _engine_seed(seed)
    if case["start"] == "hot":
        s = torch.where(_draws(n, 0, 0, 1, key) < 2 ** 31, 1, -1).to(torch.int8)
    else:
        s = torch.ones(n, dtype=torch.int8, device="cuda")
    grid = [L] * dims
    row = torch.arange(rows, device="cuda")
    parity = (row % L + row // L) & 1
    side = [((c + parity) & 1).bool()[:, None] for c in (0, 1)]
    thr = None if rule == "demon" else _thresholds(case)
    demons = []
    if rule == "demon":
        q = torch.from_numpy(_demons(n, seed)).cuda().reshape(rows, W, 2)
        demons = [torch.where(p, q[..., 1], q[..., 0]).to(torch.int8) for p in side]
    records = []
    for t in range(case["sweeps"]):
        for c in (0, 1):
            full = s.reshape(grid)
            h = sum(torch.roll(full, k, a) for a in range(dims) for k in (1, -1))
            pick = [v.reshape(rows, W, 2) for v in (full, h)]
            own, h = (torch.where(side[c], v[..., 1], v[..., 0]) for v in pick)
            d = dims - own * h // 2
            if rule == "demon":
                left = demons[c] - (dims - d)
                ok = (left >= 0) & (left <= QMAX)
                demons[c] = torch.where(ok, left, demons[c])
                own = torch.where(ok, -own, own)
            for m in range(case["hits"] if rule != "demon" else 0):
                u = _draws(n // 2, t, c + 2 * m, 0, key).reshape(rows, W)
                ok = u < thr[d.long()]
                d = torch.where(ok, 2 * dims - d, d)
                own = torch.where(ok, -own, own)
            both = s.reshape(rows, W, 2)
            s = torch.stack([torch.where(side[c], both[..., 0], own),
                             torch.where(side[c], own, both[..., 1])], dim=2).reshape(-1)
        demons = [torch.roll(q, 1, 0) for q in demons]
        if (t + 1) % case["every"] == 0:
            full = s.reshape(grid)
            e = sum(int((full * torch.roll(full, 1, a)).sum(dtype=torch.int64))
                    for a in range(dims))
            records.append((-e, int(s.sum(dtype=torch.int64))))
    return {"records": np.array(records, dtype=np.int64).reshape(-1, 2), "spins": s.cpu()}


def _exact_media(case, keys):
    dims, L = case["dims"], case["L"]
    n = L ** dims
    limit = min(int(Decimal(case["porosity"]) * 2 ** 32), MASK)
    pores = torch.stack([_draws(n, 0, 0, 3, k) <= limit for k in keys])
    pores = pores.reshape([len(keys)] + [L] * dims)
    C = torch.zeros_like(pores)
    if case["source"] == "face":
        C[:, 0] = pores[:, 0]
    else:
        at = (slice(None),) + (L // 2,) * dims
        C[at] = pores[at]
    steps = torch.zeros(len(keys), dtype=torch.int64, device="cuda")
    axes = tuple(range(1, dims + 1))
    while True:
        N = C.clone()
        for a in axes:
            N.narrow(a, 1, L - 1).logical_or_(C.narrow(a, 0, L - 1))
            N.narrow(a, 0, L - 1).logical_or_(C.narrow(a, 1, L - 1))
        N &= pores
        grew = (N != C).flatten(1).any(1)
        if not bool(grew.any()):
            break
        steps += grew
        C = N
    spans = C[:, 0].flatten(1).any(1) & C[:, L - 1].flatten(1).any(1)
    return C, C.flatten(1).sum(1), spans.to(torch.int64), steps


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return _exact_lattice(case, seed)
    if kind == "medium":
        C, size, spans, steps = _exact_media(case, [_engine_seed(seed)])
        return {"size": int(size), "spans": int(spans), "steps": int(steps),
                "cluster": C.reshape(-1).to(torch.uint8).cpu()}
    if kind == "media" and case["media"] * case["L"] ** case["dims"] <= 1 << 26:
        C, size, spans, steps = _exact_media(case, [int(k) for k in _media_seeds(case, seed)])
        return {"results": torch.stack([size, spans, steps], dim=1).cpu(),
                "clusters": C.reshape(-1).to(torch.uint8).cpu()}
    return None  # hundreds of lattices one after another would take minutes
