"""What surrounds the generations (and the sampler entry point): the prefix sums of the primaries' budgets
(blocks of 256 primaries each, up to 304 blocks and then longer ranges), and
tallies accumulated in the caller's buffers or copied to them."""
import dataclasses

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gvmod():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    return gv


@pytest.mark.parametrize("n", [1, 255, 256, 257, 304 * 256, 304 * 256 + 1, 100_003])
def test_budget_sums_admit_every_primary(gvmod, n):
    """Uneven photons through a queue that holds a few hundred of them at a
    time: the automatic cap reads the budget sums at every generation, admits
    all primaries and never overflows, and the results are those of a queue
    that holds all at once."""
    wl = W.photon_slab(n, 0.3)
    wl.primaries["E"] = 0.05 + 0.9 * np.random.default_rng(n).random(n)
    runs = []
    for cap in (1 << 16, 1 << 24):
        ctx = gvmod.Context(wl, gvmod.gv_default_config(stack_capacity=cap, per_event_counts=1))
        runs.append(ctx.transport(per_event=True))
        ctx.close()
        assert runs[-1]["status"] == 0
        assert runs[-1]["counters"]["live_peak"] <= cap
    assert np.array_equal(runs[0]["counts"][:, :11], runs[1]["counts"][:, :11])
    assert runs[0]["counters"]["tracks_gamma"] == n
    if n > 2048:  # 64 budgeted tracks each and a little: about a thousand photons in flight
        assert runs[0]["counters"]["live_peak"] <= 1024
    total = runs[0]["edep"].sum(1) + runs[0]["escape"]
    assert np.abs(total - wl.primaries["E"]).max() < 1e-6


@pytest.mark.parametrize("where", ["device", "pinned", "pageable", "unaligned"])
def test_tallies_in_place_or_copied(gvmod, where):
    import torch
    wl = W.wsi_cells(5, 3000.0)
    ctx = gvmod.Context(wl, gvmod.gv_default_config(stack_capacity=1 << 18, per_event_counts=1))
    ref = ctx.transport(per_event=True)
    shapes = {"edep": (5, ctx.n_subtotal), "escape": (5,), "cell": (50 * 32 * 32,), "counts": (5, gvmod.NCOUNT)}
    buf = {}
    for k, shape in shapes.items():
        dtype = torch.int64 if k == "counts" else torch.float64
        if where == "unaligned":  # 4 bytes off: copied, not accumulated in place
            raw = torch.full((8 * int(np.prod(shape)) + 8,), 7, dtype=torch.uint8, device="cuda")
            buf[k] = raw[4:-4]
        else:
            buf[k] = torch.full(shape, 7, dtype=dtype, device="cuda" if where == "device" else "cpu")
            if where == "pinned":
                buf[k] = buf[k].pin_memory()
    for _ in range(2):  # the second call starts from the first one's results
        ctx.gv_transport(wl.primaries, 5, wl.seed, buf["edep"], buf["cell"], buf["escape"], buf["counts"])
    torch.cuda.synchronize()
    got = {k: v.cpu().numpy().copy().view(np.int64 if k == "counts" else np.float64).reshape(shapes[k])
           for k, v in buf.items()}
    ctx.close()
    assert np.array_equal(got["counts"][:, :11], ref["counts"][:, :11])
    for k in ("edep", "escape", "cell"):  # the order of the FP64 sums
        assert np.abs(got[k].ravel() - ref[k].ravel()).max() < 1e-9 * 3000.0, k


@pytest.mark.parametrize("model", range(6))
def test_sampler_kernels_agree_at_their_border(gvmod, model):
    """From 2^20 samples on the sampling tables are read from shared memory:
    the same tables and arithmetic in another kernel, so equal up to the
    rounding of separately compiled FP32 code (a few ulp), except where that
    decides a table bin (bounded at 1e-4 of the samples)."""
    import torch
    border = 1 << 20
    wl = W.pbps_electrons(1)
    ctx = gvmod.Context(wl, gvmod.gv_default_config(stack_capacity=1 << 12))
    n = border + 77
    lo = [0.01, 2.0, 1.5, 3.0, 2.0, 0.01][model]
    E = torch.from_numpy(lo * 10.0 ** (4.0 * np.random.default_rng(model).random(n))).cuda()
    outs = []
    for m in (border - 1, border, n):
        out = torch.full((n, 3), -7.0, dtype=torch.float64, device="cuda")
        ctx.gv_unit_sample(model, 0, E[:m], 99, out)
        outs.append(out.cpu().numpy())
        assert (outs[-1][m:] == -7.0).all()
        assert (outs[-1][:m, 2] == 1.0).all()
    ctx.close()
    assert np.array_equal(outs[1][:border], outs[2][:border])
    a, b = outs[0][:border - 1], outs[1][:border - 1]
    off = np.abs(a - b) > 1e-6 * np.maximum(np.abs(a), 1e-30)
    assert off.any(axis=1).mean() < 1e-4


@pytest.mark.parametrize("integral", [False, True])
@pytest.mark.parametrize("n_layers", [2, 100, 128])
def test_histories_do_not_depend_on_where_the_integral_bound_lies(gvmod, integral, n_layers):
    """With four materials and 800 sub-slabs the bound's place in shared memory
    costs a block, and it is read from global memory; without the block stack
    there is room, and with two layers there always is: the same numbers, so
    equal counts, and deposits up to the order of their FP64 sums."""
    wl = W.pbps_electrons(200, 500.0)
    wl = dataclasses.replace(wl, materials=[W.LEAD, W.POLYSTYRENE, W.TUNGSTEN, W.SILICON], n_layers=n_layers,
                             sub_thick=[0.05, 0.2, 0.02, 0.1, 0.05, 0.1, 0.03, 0.05], sub_mat=[0, 1, 2, 3, 0, 1, 2, 3])
    if integral:
        wl = W.with_integral(wl)
    out = []
    for kw in (dict(), dict(local_stack=0), dict(block_size=64)):
        ctx = gvmod.Context(wl, gvmod.gv_default_config(per_event_counts=1, stack_capacity=1 << 18, **kw))
        out.append(ctx.transport(per_event=True))
        ctx.close()
        assert out[-1]["status"] == 0
    for r in out[1:]:
        assert np.array_equal(r["counts"][:, :11], out[0]["counts"][:, :11])
        assert np.abs(r["edep"] - out[0]["edep"]).max() < 1e-9 * 500.0
