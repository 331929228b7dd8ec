"""Boxes whose lateral walls are nearer than the planes ahead, where a bound to
the nearest wall clears hardly any step: histories do not depend on how steps
are cut into runs, and tracks take their whole budget of steps there, too."""
import dataclasses
import os

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _narrow(n=150):
    """A homogeneous bar, 1 x 1 cm and 10 cm long, hit by all three kinds."""
    wl = W.pbps_electrons(n, 200.0)
    p = wl.primaries
    p["type"] = np.arange(n) % 3
    p["x"], p["y"] = np.random.default_rng(3).uniform(-0.49, 0.49, (2, n))
    return dataclasses.replace(wl, n_layers=1, materials=[W.POLYSTYRENE], sub_thick=[10.0], sub_mat=[0], half_x=0.5,
                               half_y=0.5)


LAYOUTS = {
    "bar": _narrow,
    "slabs": lambda: dataclasses.replace(_narrow(), n_layers=20, sub_thick=[0.2, 0.3], sub_mat=[0, 0], half_x=0.05, half_y=0.5),
    "bar-field": lambda: W.with_field(_narrow(), 4.0, 0),
    "bar-msc": lambda: W.with_msc(_narrow()),
}


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
def test_histories_beside_a_wall_do_not_depend_on_the_run_length(oracle_mod, layout, prec):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = LAYOUTS[layout]()
    wl.primaries["x"] = np.clip(wl.primaries["x"], -0.98 * wl.half_x, 0.98 * wl.half_x)
    runs = []
    for budget in (1, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, per_event_counts=1, stack_capacity=1 << 18,
                                                  along_steps=budget, along_steps_photon=budget, tail_threshold=0))
        runs.append(ctx.transport(per_event=True))
        ctx.close()
        assert runs[-1]["status"] == 0
    one, many = runs
    assert np.array_equal(one["counts"][:, :11], many["counts"][:, :11])
    assert np.abs(one["edep"] - many["edep"]).max() < 1e-9 * 200.0
    assert np.abs(one["escape"] - many["escape"]).max() < 1e-9 * 200.0
    if prec:
        ref = oracle_mod.Oracle(wl).transport(n_threads=os.cpu_count() or 4)
        same = np.all(many["counts"][:, :11] == ref["counts"][:, :11], axis=1)
        assert same.mean() >= 0.9, same.mean()
        assert np.abs(many["edep"][same] - ref["edep"][same]).max() < 1e-9 * 200.0


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("sort", [dict(), dict(pipeline=1)], ids=["sort", "split"])
def test_charged_runs_go_on_beside_a_wall(oracle_mod, prec, sort):
    """Electrons that only lose energy continuously, half a centimetre from the
    walls: with one round a generation, and budgets of one step and of 64, the
    generations are the steps of the longest track, and one or two runs."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = dataclasses.replace(_narrow(64), process_mask=W.P_IONI, e_cut=1e30)
    wl.primaries["type"] = W.ELECTRON
    wl.primaries["E"] = 10.0
    gens = []
    for budget in (1, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, stack_capacity=1 << 12, along_steps=budget,
                                                  tail_threshold=0, **sort))
        r = ctx.transport()
        ctx.close()
        assert r["status"] == 0
        gens.append(r["counters"]["generations"])
    longest = oracle_mod.Oracle(wl).transport(n_threads=4)["counts"][:, 0].max()
    assert 10 < longest <= 64
    assert gens[0] >= longest and gens[1] <= 2, gens


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("sort", [dict(), dict(pipeline=1)], ids=["sort", "split"])
def test_photon_runs_go_on_beside_a_wall(prec, sort):
    """Photons that do not interact, across 50 slabs of half a millimetre, 0.1 to
    0.9 mm from the walls and slowly towards them: with one round a generation
    and a budget of 64 steps they cross in one run.  Those that reach a wall
    take the last step in a second one, or a third where the first ended a step
    early: the bound is short by a thousandth of a step and 1e-4 of the path."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    n = 64
    wl = dataclasses.replace(_narrow(n), n_layers=50, sub_thick=[0.05], half_x=0.1, half_y=0.1, process_mask=W.P_PAIR)
    p = wl.primaries
    p["type"], p["E"] = W.GAMMA, 0.9
    p["x"], p["y"] = np.linspace(0.01, 0.09, n), -np.linspace(0.09, 0.01, n)
    p["u"], p["v"] = np.linspace(0.0, 0.03, n), -np.linspace(0.03, 0.0, n)
    p["w"] = np.sqrt(1.0 - p["u"] ** 2 - p["v"] ** 2)
    gens, escaped = [], []
    for budget in (1, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, stack_capacity=1 << 12, along_steps_photon=budget,
                                                  tail_threshold=0, **sort))
        r = ctx.transport()
        ctx.close()
        assert r["status"] == 0
        gens.append(r["counters"]["generations"])
        escaped.append((r["counters"]["steps"], r["counters"]["unscattered"], r["escape"].tolist()))
    assert escaped[0] == escaped[1] and 0 < escaped[0][1] < n  # some leave through the far plane, some through a wall
    assert gens[0] >= 50 and gens[1] <= 3, gens
