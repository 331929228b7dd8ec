"""Runs of along-steps: a track's history does not depend on how its steps
are cut into runs, whichever way it crosses the planes.  Photons that entered
a sub-slab in their own run take its thickness from a table instead of
subtracting coordinates, so backward, oblique, lateral and on-plane starts are
run with one step per run (every distance from coordinates) and with long
runs.  With one step per run against many the same FP32 operations are done:
integer counts are equal and deposits differ by the order of the FP64 sums."""
import dataclasses
import os

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _both_ways(n=96):
    wl = W.pbps_electrons(n, 400.0)
    p = wl.primaries
    rng = np.random.default_rng(5)
    p["type"] = np.arange(n) % 3
    p["z"] = np.where(np.arange(n) % 2, 0.7 * rng.integers(0, 50, n), rng.uniform(0.0, 35.0, n))
    c = rng.uniform(-1.0, 1.0, n)
    c[:4] = (1.0, -1.0, 0.0, 1e-3)  # along the axis both ways, lateral, grazing
    phi = rng.uniform(0.0, 2.0 * np.pi, n)
    s = np.sqrt(1.0 - c * c)
    p["u"], p["v"], p["w"] = s * np.cos(phi), s * np.sin(phi), c
    p["x"], p["y"] = rng.uniform(-19.9, 19.9, (2, n))
    return wl


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
def test_histories_do_not_depend_on_the_run_length(oracle_mod, prec):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = _both_ways()
    runs = []
    for budget in (1, 2, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, per_event_counts=1, stack_capacity=1 << 20,
                                                  along_steps=budget, along_steps_photon=budget))
        runs.append(ctx.transport(per_event=True))
        ctx.close()
        assert runs[-1]["status"] == 0
    base = runs[0]
    for r in runs[1:]:
        assert np.array_equal(r["counts"][:, :11], base["counts"][:, :11])
        assert np.abs(r["edep"] - base["edep"]).max() < 1e-9 * 400.0
        assert np.abs(r["escape"] - base["escape"]).max() < 1e-9 * 400.0
    if prec:  # and the histories are the oracle's
        ref = oracle_mod.Oracle(wl).transport(n_threads=os.cpu_count() or 4)
        same = np.all(base["counts"][:, :11] == ref["counts"][:, :11], axis=1)
        assert same.mean() >= 0.9, same.mean()
        assert np.abs(base["edep"][same] - ref["edep"][same]).max() < 1e-9 * 400.0


@pytest.mark.parametrize("cap", [3, 0], ids=["3-in-flight", "no-cap"])
def test_event_bookkeeping_follows_the_in_flight_cap(cap):
    """An event's live tracks are booked only while primaries wait on the
    cap; whether they are must not change a history, and a cap of three
    events with three primaries each must still let every event through."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.pbps_electrons(45, 300.0)
    wl.primaries["event"] = np.arange(45) // 3
    wl.primaries["id"] = np.arange(45) % 3
    wl.primaries["type"] = np.arange(45) % 3
    wl.n_events = 15
    out = []
    for kw in (dict(), dict(max_events_in_flight=cap, refill_batch=4), dict(pipeline=1, max_events_in_flight=cap),
               dict(process_sort=0, max_events_in_flight=cap)):
        ctx = gv.Context(wl, gv.gv_default_config(per_event_counts=1, stack_capacity=1 << 18, **kw))
        out.append(ctx.transport(per_event=True))
        ctx.close()
        assert out[-1]["status"] == 0, kw
        assert np.array_equal(out[-1]["counts"][:, :11], out[0]["counts"][:, :11]), kw
    if cap:  # three events in flight take many more generations than all at once
        assert out[1]["counters"]["generations"] > 2 * out[0]["counters"]["generations"]


@pytest.mark.parametrize("precision", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("tesla", [1e-12, 1e-34, 1e-37, 1e-40])
def test_field_too_weak_to_turn_a_step(precision, tesla):
    """Turns down to the subnormal numbers and zero: the step is the straight
    one (its own rounding, three products and two sums: 5 half-ulps; and the
    turn itself, 0.29 / cm of a 10 MeV track in 1 T, where it is a number)."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.with_field(W.pbps_electrons(1), tesla, 1)
    ctx = gv.Context(wl, gv.gv_default_config(precision=precision, stack_capacity=1 << 12))
    n = 64
    s = np.repeat(10.0 ** np.arange(-14.0, 2.0), 4)
    d = np.tile([[0.6, 0.0, 0.8], [0.0, 1.0, 0.0], [0.48, 0.6, -0.64], [0.0, 0.0, 1.0]], (n // 4, 1))
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    out = torch.zeros((n, 7), dtype=torch.float64, device="cuda")
    ctx.gv_unit_field(1, dev(np.full(n, 10.0)), dev(s), dev(d), out)
    g = out.cpu().numpy()
    ctx.close()
    eps = 2.0 ** (-22 if precision == 0 else -51)
    assert (np.abs(g[:, :3] - s[:, None] * d) <= eps * s[:, None] + tesla * s[:, None] ** 2).all()
    assert (np.abs(g[:, 3:6] - d) <= eps + tesla * s[:, None]).all()


@pytest.mark.parametrize("thick, mat", [([0.2, 0.2, 0.5], [0, 1, 0]), ([0.3, 0.1, 0.1], [0, 0, 1]), ([0.4], [1])])
def test_fp64_runs_across_repeated_slabs(thick, mat):
    """An FP64 photon run takes cross sections and paths over from the
    sub-slab before the last where table row or thickness are the same: each
    may repeat without the other, and in a stack of one kind always.  One step
    a run takes nothing over, and gives the same histories."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = dataclasses.replace(_both_ways(), n_layers=50, sub_thick=thick, sub_mat=mat)
    out = []
    for budget in (1, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=1, per_event_counts=1, stack_capacity=1 << 20,
                                                  along_steps=budget, along_steps_photon=budget))
        out.append(ctx.transport(per_event=True))
        ctx.close()
        assert out[-1]["status"] == 0
    assert np.array_equal(out[0]["counts"][:, :11], out[1]["counts"][:, :11])
    assert np.abs(out[0]["edep"] - out[1]["edep"]).max() < 1e-9 * 400.0
    assert np.abs(out[0]["escape"] - out[1]["escape"]).max() < 1e-9 * 400.0


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("block", [64, 256])
def test_a_full_block_stack_loses_no_secondary(prec, block):
    """Blocks of charged tracks with long claims make more secondaries a round
    than their stacks hold, so reservations are refused all the time, several
    at once in the larger block: histories stay those without a stack."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.pbps_electrons(40_000 if prec == 0 else 8_000, 60.0)
    out = []
    for kw in (dict(local_stack=0, tail_steps_per_claim=1), dict(tail_steps_per_claim=16, tail_threshold=1 << 40)):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, per_event_counts=1, block_size=block,
                                                  stack_capacity=1 << 20, **kw))
        for _ in range(3):
            out.append(ctx.transport(per_event=True))
            assert out[-1]["status"] == 0, kw
            assert np.array_equal(out[-1]["counts"][:, :11], out[0]["counts"][:, :11]), kw
            assert np.abs(out[-1]["edep"] - out[0]["edep"]).max() < 1e-9 * 60.0, kw
        ctx.close()
