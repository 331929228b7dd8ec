"""A step in a magnetic field that ends on a lateral wall: the wall is the one
the pre-step direction points at, also where the field turns the track away
from it within the step.  Positrons just above the tracking cut graze a wall
and stop on it, so the two photons of their annihilation start there.  And the
field's own step limit, down to curvatures below the FP32 normal range."""
import dataclasses
import os

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _grazing(axis, n=256):
    """Field along `axis` (0 x, 1 y): tracks along +-z next to the walls of the
    other lateral axis, 60 to 100 um from them along their path.  At 0.3 MeV
    the field turns them by 0.11 to 0.19 rad on the way, their angle to the
    wall is 0.02 to 0.08 rad, and they lose 13 keV or more of the 5 keV that
    they have above the cut."""
    wl = W.with_field(W.pbps_electrons(n, 0.305), 4.0, axis)
    wl = dataclasses.replace(wl, track_cut=0.3)
    p = wl.primaries
    rng = np.random.default_rng(17 + axis)
    side = np.where(np.arange(n) % 2, 1.0, -1.0)
    fwd = np.where(np.arange(n) // 2 % 2, 1.0, -1.0)
    angle, path = rng.uniform(0.02, 0.08, n), rng.uniform(0.006, 0.010, n)
    p["type"] = W.POSITRON
    p["z"] = 0.7 * rng.integers(0, 50, n) + 0.2 + rng.uniform(0.1, 0.4, n)  # inside a polystyrene sub-slab
    p["w"] = fwd * np.cos(angle)
    near, other = ("y", "x") if axis == 0 else ("x", "y")
    p[near] = side * (20.0 - np.sin(angle) * path)
    p[other] = rng.uniform(-10.0, 10.0, n)
    p["v" if axis == 0 else "u"] = side * np.sin(angle)
    return wl


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("sort", [0, 1], ids=["no-sort", "sort"])
def test_track_turned_away_stops_on_its_wall(oracle_mod, axis, prec, sort):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = _grazing(axis)
    ref = oracle_mod.Oracle(wl).transport(n_threads=os.cpu_count() or 4)
    ctx = gv.Context(wl, gv.gv_default_config(precision=prec, per_event_counts=1, stack_capacity=1 << 14,
                                              process_sort=sort))
    r = ctx.transport(per_event=True)
    ctx.close()
    assert r["status"] == 0
    # one positron step, one annihilation (a few annihilate in flight)
    assert (ref["counts"][:, 3] == 1).mean() > 0.95 and (ref["counts"][:, 8] == 1).mean() > 0.95
    # the histories are the oracle's: in FP64 but for knife-edge decisions, in
    # FP32 but for a few where rounding moves a decision of a photon's history
    same = np.all(r["counts"][:, :11] == ref["counts"][:, :11], axis=1)
    assert same.mean() >= (0.98 if prec else 0.9), same.mean()
    tol = 1e-9 if prec else 1e-4
    assert np.abs(r["edep"][same] - ref["edep"][same]).max() < tol
    assert np.abs(r["escape"][same] - ref["escape"][same]).max() < tol


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("tesla", [4.0, 1e-12, 1e-36, 1e-38, 1e-39, 1e-40])
def test_step_limit_of_the_weakest_fields(oracle_mod, prec, tesla):
    """The limit is the square root of a quotient by the curvature: finite
    where that quotient is, although the curvature's reciprocal is not.  A
    curvature below 1.2e-38 / cm holds multiples of 2^-149; it is rounded
    three times on the way (constant, quotient by p, sine)."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.with_field(W.pbps_electrons(1), tesla, 1)
    ctx = gv.Context(wl, gv.gv_default_config(precision=prec, stack_capacity=1 << 12))
    o = oracle_mod.Oracle(wl)
    E = np.array([0.1, 1.0, 10.0, 30.0])
    d = np.tile([[0.6, 0.0, 0.8]], (4, 1))
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    out = torch.zeros((4, 7), dtype=torch.float64, device="cuda")
    ctx.gv_unit_field(1, dev(E), dev(np.full(4, 0.1)), dev(d), out)
    got = out.cpu().numpy()[:, 6]
    ctx.close()
    for i in range(4):
        want = o.field_step_limit(1, E[i], d[i])
        curv = 2.99792458 * tesla / np.sqrt(E[i] * (E[i] + 2 * 0.51099895))
        tol = 1e-5 + 3 * 2.0 ** -149 / curv if prec == 0 else 1e-12
        if prec == 0 and want ** 2 > 3.4028235e38:  # the quotient overflows, as a division's does
            assert got[i] == np.inf
            continue
        assert abs(got[i] - want) <= tol * want, (E[i], got[i], want)
