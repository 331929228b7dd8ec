"""gv_transport_static on the basketizing kernel: over the configurations that
shape its launch it gives the showers of a context without the basketizer
(the arithmetic it keeps), deposits up to the order of the FP64 sums."""
import ctypes as C

import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _static(gv, ctx, wl):
    import torch
    prim = torch.from_numpy(wl.primaries.view(np.uint8).copy()).cuda()
    edep = torch.full((wl.n_events, ctx.n_subtotal), 7.0, dtype=torch.float64, device="cuda")
    esc = torch.full((wl.n_events,), 7.0, dtype=torch.float64, device="cuda")
    counters = (C.c_ulonglong * 16)()
    rc = ctx.lib.gv_transport_static(ctx.h, prim.data_ptr() if len(wl.primaries) else None, len(wl.primaries),
                                     wl.n_events, C.c_ulonglong(wl.seed), torch.cuda.current_stream().cuda_stream,
                                     edep.data_ptr(), esc.data_ptr(), counters)
    assert rc == 0, gv.load().gv_strerror(rc)
    return edep.cpu().numpy(), esc.cpu().numpy(), list(counters)


@pytest.mark.parametrize("options", ["plain", "msc", "rejection", "integral"])
@pytest.mark.parametrize("config", [dict(), dict(block_size=64), dict(block_size=96, local_stack=0),
                                    dict(pipeline=1), dict(process_sort=0, block_size=128),
                                    dict(tail_threshold=0, pdl=0)],
                         ids=["default", "64", "96-no-stack", "split-context", "plain-context", "no-tail"])
def test_static_matches_the_plain_kernel(options, config):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.pbps_mixed(37)
    wl.primaries["E"] = np.minimum(wl.primaries["E"], 2000.0)
    wl = {"plain": lambda w: w, "msc": W.with_msc, "rejection": W.with_rejection, "integral": W.with_integral}[options](wl)
    plain = gv.Context(wl, gv.gv_default_config(stack_capacity=1 << 20, process_sort=0, claim_chunks=0))
    ref = plain.transport()
    plain.close()
    ctx = gv.Context(wl, gv.gv_default_config(stack_capacity=1 << 16, **config))
    for _ in range(2):  # the second call starts from what the first left in the scratch array
        edep, esc, cnt = _static(gv, ctx, wl)
    ctx.close()
    for i in range(11):
        assert cnt[i] == ref["counters"][gv.COUNTER_NAMES[i]], gv.COUNTER_NAMES[i]
    scale = np.maximum(ref["edep"].sum(1, keepdims=True), 1.0)
    assert (np.abs(edep - ref["edep"]) / scale).max() < 1e-9
    assert np.abs(esc - ref["escape"]).max() < 1e-9 * max(1.0, ref["escape"].max())


def test_static_without_primaries():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    import dataclasses
    wl = W.pbps_electrons(3, 100.0)
    ctx = gv.Context(wl, gv.gv_default_config(stack_capacity=1 << 16))
    edep, esc, cnt = _static(gv, ctx, dataclasses.replace(wl, primaries=wl.primaries[:0]))
    ctx.close()
    assert not edep.any() and not esc.any() and cnt[0] == 0
