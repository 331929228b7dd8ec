"""The integral approach rejects most interactions of slow positrons (the bound
follows the annihilation cross section at the lowest energies): a run of steps
goes on through them, and the histories stay the same."""
import dataclasses
import os

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("kw", [dict(), dict(pipeline=1)], ids=["sort", "split"])
def test_runs_go_on_through_rejected_interactions(oracle_mod, prec, kw):
    """With one round a generation, a positron of `longest` steps needs a
    generation for every 64 of them with a budget of 64; its annihilation and
    the photons' flight out of the box (two runs) come after."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    n = 96
    wl = W.with_integral(dataclasses.replace(W.pbps_electrons(n, 10.0), n_layers=1, materials=[W.POLYSTYRENE],
                                             sub_thick=[20.0], sub_mat=[0], process_mask=W.P_ANNIH, e_cut=1e30))
    wl.primaries["type"] = W.POSITRON
    wl.primaries["E"] = np.linspace(0.05, 10.0, n)
    wl.primaries["z"] = 5.0
    ref = oracle_mod.Oracle(wl).transport(n_threads=os.cpu_count() or 4)
    longest = int(ref["counts"][:, 3].max())
    gens = []
    for budget in (1, 64):
        ctx = gv.Context(wl, gv.gv_default_config(precision=prec, per_event_counts=1, stack_capacity=1 << 14,
                                                  along_steps=budget, along_steps_photon=budget, tail_threshold=0, **kw))
        r = ctx.transport(per_event=True)
        ctx.close()
        assert r["status"] == 0
        same = np.all(r["counts"][:, :11] == ref["counts"][:, :11], axis=1)
        assert same.mean() >= (0.98 if prec else 0.9), same.mean()
        assert np.abs(r["edep"][same] - ref["edep"][same]).max() < (1e-9 if prec else 1e-4) * 10.0
        gens.append(r["counters"]["generations"])
    assert longest > 20
    assert gens[0] >= longest and gens[1] <= -(-longest // 64) + 3, (longest, gens)
