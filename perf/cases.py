"""Performance cases: the transports a user of this library runs, through its
public entry points, over the range they are run in.

Every case but one is a whole shower transport (gv_transport or
gv_transport_static): primaries in hand, tallies and counters back.  The one
that is not samples Bethe-Heitler pairs element by element, the paper's own
sampler comparison (Sec. 3.5).

A transport's outputs are its tallies and the counters of what the tracks did
(steps, tracks, pairs, ...).  How the work was scheduled -- generations, lane
slots, peak population -- is a diagnostic of the library's own and not a
result of the transport, so those three counters are left out.
"""
import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_2005_00949_gb300 import gv, workloads as W

# counters that depend on the histories only, by their place in gv_result.counters
PHYSICS_COUNTERS = (0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 13)

# track steps per MeV of primary energy (rounded, from the workloads as they
# run) and sub-slabs: what work() needs to know of each layout
LAYOUTS = {"pbps": (3.75, 100), "pblar": (5.3, 100), "wsi": (3.2, 100), "slab": (4.6, 1)}
# FP32 operations of one step and its share of an interaction: two table
# rows interpolated, limits, displacement, loss; a fifth of a final state
FLOPS_PER_STEP = 150.0


def listed():
    return [
        # one event handed over by an event loop: all latency
        {"name": "one_10GeV_shower", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 10000.0,
         "events": 1},
        # a test beam run at low energy: 1000 x 1 GeV e-, a standard workload
        {"name": "pbps_1GeV_1000", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 1000.0,
         "events": 1000},
        # the benchmark workload: 2000 x 10 GeV e- in Pb/polystyrene
        {"name": "pbps_10GeV_2000", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 10000.0,
         "events": 2000},
        # the standard mixed-type batch: e-, e+, gamma, 0.1 to 100 GeV
        {"name": "pbps_mixed_4096", "kind": "transport", "layout": "pbps", "beam": "mixed", "energy": 100000.0,
         "events": 4096},
        # high-granularity calorimeter with its cell histogram (the standard
        # W/Si workload, 2000 of its events)
        {"name": "wsi_100GeV_cells_2000", "kind": "transport", "layout": "wsi", "beam": "e-", "energy": 100000.0,
         "events": 2000},
        # the paper's TestEm3 conditions: Pb/LAr, 4 T, multiple scattering
        {"name": "testem3_4T_msc_1000", "kind": "transport", "layout": "pblar", "beam": "e-", "energy": 10000.0,
         "events": 1000, "msc": True, "field": 4.0},
        # the same layout without the options, host buffers in and out: what a
        # program without device memory of its own calls
        {"name": "testem3_host_buffers_1000", "kind": "transport", "layout": "pblar", "beam": "e-", "energy": 10000.0,
         "events": 1000, "host": True},
        # FP64 everywhere: the validation runs
        {"name": "pbps_fp64_10GeV_300", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 10000.0,
         "events": 300, "fp64": True},
        # several primaries per event (the paper's events hold sixteen
        # electrons) with counters kept per event; a ragged number of events
        {"name": "pbps_16x1GeV_counts_61", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 1000.0,
         "events": 61, "per_event": 16, "counts": True},
        # photon transmission through a thick slab (standard workload)
        {"name": "slab_1MeV_photons_1e5", "kind": "transport", "layout": "slab", "beam": "gamma", "energy": 1.0,
         "events": 100000},
        # a host framework that owns the GPU's memory: no allocation
        {"name": "static_10GeV_37", "kind": "transport", "layout": "pbps", "beam": "e-", "energy": 10000.0,
         "events": 37, "static": True},
        # the paper's pair-sampler comparison, sampling tables
        {"name": "pair_tables_4M", "kind": "sampler", "n": 4 << 20},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges: any layout with the options it is
    run with, 0.5 to 100 GeV per primary, one event to thousands, up to a
    total energy that keeps the case below the largest listed one."""
    kind = rng.choice(["pbps", "pbps", "pbps", "mixed", "wsi", "pblar", "pblar", "slab", "static", "sampler"])
    if kind == "sampler":
        return {"kind": "sampler", "n": int(_log_uniform(rng, 1000, 4 << 20))}
    if kind == "slab":
        return {"kind": "transport", "layout": "slab", "beam": "gamma",
                "energy": round(_log_uniform(rng, 0.2, 5.0), 3), "events": int(_log_uniform(rng, 100, 200000))}
    if kind == "mixed":
        return {"kind": "transport", "layout": "pbps", "beam": "mixed", "energy": 100000.0,
                "events": int(_log_uniform(rng, 10, 4096))}
    if kind == "static":
        energy = round(_log_uniform(rng, 500.0, 20000.0), 1)
        return {"kind": "transport", "layout": "pbps", "beam": rng.choice(["e-", "e+", "gamma"]), "energy": energy,
                "events": int(_log_uniform(rng, 1, 400000.0 / energy)), "static": True}
    energy = round(_log_uniform(rng, 500.0, 100000.0), 1)
    case = {"kind": "transport", "layout": kind, "beam": rng.choice(["e-", "e-", "e+", "gamma"]), "energy": energy}
    total = {"pbps": 2.0e7, "wsi": 1.0e8, "pblar": 1.0e7}[kind]
    if kind == "pblar":
        if rng.random() < 0.6:
            case["msc"] = True
            if rng.random() < 0.7:
                case["field"] = 4.0
        elif rng.random() < 0.5:
            case["host"] = True
    if kind == "pbps":
        if rng.random() < 0.25:
            case["fp64"] = True
            total = 3.0e6
        if rng.random() < 0.25:
            case["counts"] = True
        if rng.random() < 0.25:
            case["per_event"] = rng.choice([2, 3, 16])
    per_event = case.get("per_event", 1)
    case["events"] = max(1, int(_log_uniform(rng, 1, max(2.0, min(4000.0, total / (energy * per_event))))))
    return case


def _workload(case, seed):
    rng = np.random.default_rng([seed, 20])
    n_events, per_event = case["events"], case.get("per_event", 1)
    n = n_events * per_event
    layout, energy = case["layout"], case["energy"]
    if layout == "slab":
        wl = W.photon_slab(n, energy)
    elif layout == "wsi":
        wl = W.wsi_cells(n, energy)
    elif layout == "pblar":
        wl = W.pblar_testem3(n, energy)
    else:
        wl = W.pbps_electrons(n, energy)
    p = wl.primaries
    p["event"] = np.arange(n) // per_event
    p["id"] = np.arange(n) % per_event
    if case["beam"] == "mixed":
        p["type"] = p["event"] % 3
        p["E"] = 100.0 * (energy / 100.0) ** rng.random(n)
    else:
        p["type"] = {"gamma": W.GAMMA, "e-": W.ELECTRON, "e+": W.POSITRON}[case["beam"]]
    spread = 2.5 if layout == "wsi" else 0.1  # the central 4 x 4 cells; a beam spot of 2 mm
    p["x"] = rng.uniform(-spread, spread, n)
    p["y"] = rng.uniform(-spread, spread, n)
    if case.get("msc"):
        wl = W.with_msc(wl)
    if case.get("field"):
        wl = W.with_field(wl, case["field"])
    return dataclasses.replace(wl, n_events=n_events, seed=int(rng.integers(1 << 62)))


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "sampler":
        rng = np.random.default_rng([seed, 21])
        ctx = gv.Context(W.pbps_electrons(1), gv.gv_default_config(stack_capacity=1 << 12))
        energy = 2.0 * (1e5 / 2.0) ** rng.random(case["n"])  # 2 MeV to 100 GeV
        return {"kind": "sampler", "ctx": ctx, "energy": torch.from_numpy(energy).to(dev),
                "seed": int(rng.integers(1 << 62)),
                "out": torch.empty((case["n"], 3), dtype=torch.float64, device=dev)}
    wl = _workload(case, seed)
    config = gv.gv_default_config(precision=gv.GV_FP64 if case.get("fp64") else gv.GV_MIXED,
                                  per_event_counts=1 if case.get("counts") else 0)
    ctx = gv.Context(wl, config)
    n, nsub = wl.n_events, ctx.n_subtotal
    prim = torch.from_numpy(wl.primaries.view(np.uint8).copy())
    edep = torch.zeros((n, nsub), dtype=torch.float64)
    escape = torch.zeros(n, dtype=torch.float64)
    if case.get("host"):
        prim, edep, escape = prim.pin_memory(), edep.pin_memory(), escape.pin_memory()
    else:
        prim, edep, escape = prim.to(dev), edep.to(dev), escape.to(dev)
    ncell = wl.n_layers * wl.nx * wl.ny
    return {"kind": "static" if case.get("static") else "transport", "ctx": ctx, "wl": wl, "prim": prim,
            "edep": edep, "escape": escape,
            "cell": torch.zeros(ncell, dtype=torch.float64, device=dev) if ncell else None,
            "counts": torch.zeros((n, gv.NCOUNT), dtype=torch.int64, device=dev) if case.get("counts") else None}


def run(state):
    ctx = state["ctx"]
    if state["kind"] == "sampler":
        ctx.gv_unit_sample(W_PAIR, 0, state["energy"], state["seed"], state["out"])
        return state["out"]
    wl = state["wl"]
    out = {"edep": state["edep"], "escape": state["escape"]}
    if state["kind"] == "static":
        counters = (ctypes.c_ulonglong * 16)()
        rc = ctx.lib.gv_transport_static(ctx.h, state["prim"].data_ptr(), len(wl.primaries), wl.n_events,
                                         ctypes.c_ulonglong(wl.seed), torch.cuda.current_stream().cuda_stream,
                                         state["edep"].data_ptr(), state["escape"].data_ptr(), counters)
        if rc != gv.GV_OK:
            raise gv.GvError(f"gv_transport_static: {rc}")
    else:
        # the call and its gv_sync: the counters and the status are only there after it
        counters = ctx.gv_transport(state["prim"], wl.n_events, wl.seed, state["edep"], state["cell"],
                                    state["escape"], state["counts"]).counters
        if state["cell"] is not None:
            out["cell"] = state["cell"]
        if state["counts"] is not None:
            out["counts"] = state["counts"]
    out["counters"] = np.array([counters[i] for i in PHYSICS_COUNTERS], dtype=np.int64)
    return out


def work(case):
    if case["kind"] == "sampler":
        return {"bytes": 32.0 * case["n"], "flops": 40.0 * case["n"]}  # an energy in, three numbers out
    per_mev, nsub = LAYOUTS[case["layout"]]
    n = case["events"] * case.get("per_event", 1)
    mean = case["energy"]
    if case["beam"] == "mixed":  # log-uniform from 100 MeV
        mean = (case["energy"] - 100.0) / math.log(case["energy"] / 100.0)
    nbytes = 72.0 * n + 8.0 * case["events"] * (nsub + 1)
    if case["layout"] == "wsi":
        nbytes += 8.0 * 50 * 32 * 32
    if case.get("counts"):
        nbytes += 8.0 * gv.NCOUNT * case["events"]
    return {"bytes": nbytes, "flops": FLOPS_PER_STEP * per_mev * mean * n}


# ---- the pair sampler in 64 bits ------------------------------------------------
W_PAIR = 1  # GV_M_PAIR
ELECTRON_MASS = 0.51099895  # MeV


def _philox_words(index, seed):
    """Words 0..2 of Philox4x32-10 (Salmon et al., SC'11) at counter (i_lo, i_hi, 0, 0)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [index & m32, index >> np.uint64(32), np.zeros_like(index), np.zeros_like(index)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[:3]


def _pair_tables():
    """Per grid energy (8 per decade from 1.25 MeV): the density at 65 nodes of
    the reduced variable, and Vose's alias table over the 64 bins."""
    low, per_decade, bins = 1.25, 8, 64
    n_grid = 1 + math.ceil(per_decade * math.log10(1e6 / low) - 1e-6)
    xi = np.arange(bins + 1) / bins
    pdf, keep, alias = [], [], []
    for i in range(n_grid):
        a = ELECTRON_MASS / (low * 10.0 ** (i / per_decade))
        x = a + xi * (1.0 - 2.0 * a)
        f = 1.0 - 4.0 / 3.0 * x * (1.0 - x)
        mass = 0.5 * (f[:-1] + f[1:])
        total = 0.0
        for m in mass:
            total += m
        prob = [m * bins / total for m in mass]
        q, al = [1.0] * bins, list(range(bins))
        small = [j for j in range(bins) if prob[j] < 1.0]
        large = [j for j in range(bins) if not prob[j] < 1.0]
        while small and large:
            s, l = small.pop(), large.pop()
            q[s], al[s] = prob[s], l
            prob[l] = (prob[l] + prob[s]) - 1.0
            (small if prob[l] < 1.0 else large).append(l)
        pdf.append(f)
        keep.append(q)
        alias.append(al)
    return low, per_decade, np.array(pdf), np.array(keep, dtype=np.float32).astype(np.float64), np.array(alias)


def exact(case, seed):
    """The pair sampler's outputs in 64 bits.  A transport has none: its
    outputs are sums over random histories that only its own tables define."""
    if case["kind"] != "sampler":
        return None
    rng = np.random.default_rng([seed, 21])
    energy = 2.0 * (1e5 / 2.0) ** rng.random(case["n"])
    key = int(rng.integers(1 << 62))
    words = _philox_words(np.arange(case["n"], dtype=np.uint64), key)
    ug, ub, ui = [((w >> np.uint64(8)).astype(np.float64) + 1.0) / 16777216.0 for w in words]
    low, per_decade, pdf, keep, alias = _pair_tables()
    level = np.log(energy / low) * (per_decade / math.log(10.0))
    row = np.clip(np.floor(level).astype(np.int64), 0, len(pdf) - 1)
    row = np.minimum(row + (ug < level - row), len(pdf) - 1)
    place = ub * 64.0
    b = np.minimum(place.astype(np.int64), 63)
    b = np.where(place - b < keep[row, b], b, alias[row, b])
    p0, p1 = pdf[row, b], pdf[row, b + 1]
    t = ui * (p0 + p1) / (p0 + np.sqrt(p0 * p0 + ui * (p1 * p1 - p0 * p0)))
    xi = (b + t) / 64.0
    a = ELECTRON_MASS / energy
    return np.stack([a + xi * (1.0 - 2.0 * a), xi, np.ones_like(xi)], axis=1)
