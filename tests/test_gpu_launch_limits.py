"""What contexts and threads share: the limit of a kernel's dynamic shared
memory, and the scratch array of the allocation-free call.  A context made
later, or a call on another thread, that needs less of the one must leave room
for those that need more; the other is touched by one call at a time."""
import ctypes as C
import dataclasses
import threading

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


def _large(n=60, energy=300.0):
    """Four materials and 800 sub-slabs."""
    return dataclasses.replace(W.pbps_electrons(n, energy), n_layers=100,
                               materials=[W.LEAD, W.POLYSTYRENE, W.TUNGSTEN, W.SILICON],
                               sub_thick=[0.05, 0.2, 0.02, 0.1, 0.05, 0.1, 0.03, 0.05], sub_mat=[0, 1, 2, 3, 0, 1, 2, 3])


def _small(n=60):
    """One material, two sub-slabs."""
    return dataclasses.replace(W.pbps_electrons(n, 300.0), n_layers=2, materials=[W.POLYSTYRENE], sub_thick=[5.0],
                               sub_mat=[0])


@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(process_sort=0), dict(pipeline=1)],
                         ids=["sort", "fp64", "no-sort", "split"])
def test_small_context_leaves_a_large_one_its_shared_memory(gvmod, kw):
    alone = gvmod.Context(_large(), gvmod.gv_default_config(stack_capacity=1 << 18, **kw))
    ref = alone.transport()
    alone.close()
    large = gvmod.Context(_large(), gvmod.gv_default_config(stack_capacity=1 << 18, **kw))
    small = gvmod.Context(_small(), gvmod.gv_default_config(stack_capacity=1 << 18, block_size=64, **kw))
    assert small.transport()["status"] == 0
    r = large.transport()  # its kernels are captured here
    large.close()
    small.close()
    assert r["status"] == 0
    assert [r["counters"][k] for k in gvmod.COUNTER_NAMES[:11]] == [ref["counters"][k] for k in gvmod.COUNTER_NAMES[:11]]


def test_two_threads_sample_different_models(gvmod):
    """The tables of different models have different sizes (Compton 74 KB,
    pairs 49 KB): two threads that sample one each get the samples that each
    gets alone."""
    import torch
    ctx = gvmod.Context(W.pbps_electrons(1), gvmod.gv_default_config(stack_capacity=1 << 12))
    n = 1 << 20
    energy = torch.linspace(2.0, 1e4, n, dtype=torch.float64, device="cuda")
    alone, errors = {}, []
    for model in (0, 1):
        alone[model] = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        ctx.gv_unit_sample(model, 0, energy, 99, alone[model])
    torch.cuda.synchronize()

    def sample(model):
        stream = torch.cuda.Stream()
        out = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        try:
            for _ in range(3000):
                ctx.gv_unit_sample(model, 0, energy, 99, out, stream)
        except gvmod.GvError as e:
            errors.append(str(e))
        stream.synchronize()
        if not torch.equal(out, alone[model]):
            errors.append(f"model {model}: other samples")

    threads = [threading.Thread(target=sample, args=(m,)) for m in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    ctx.close()
    assert not errors, errors


def _static_calls(gv, ctx, wl, n, out):
    import torch
    stream = torch.cuda.Stream()
    prim = torch.from_numpy(wl.primaries.view(np.uint8).copy()).cuda()
    edep = torch.zeros((wl.n_events, ctx.n_subtotal), dtype=torch.float64, device="cuda")
    esc = torch.zeros(wl.n_events, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(n):
        counters = (C.c_ulonglong * 16)()
        rc = ctx.lib.gv_transport_static(ctx.h, prim.data_ptr(), len(wl.primaries), wl.n_events,
                                         C.c_ulonglong(wl.seed), stream.cuda_stream, edep.data_ptr(), esc.data_ptr(),
                                         counters)
        stream.synchronize()
        out.append((rc, list(counters)[:11], edep.cpu().numpy(), esc.cpu().numpy()))


def test_static_calls_of_two_threads(gvmod):
    """Contexts of different sizes, driven at once: every call gives what it
    gives alone, whatever the other thread's call sets up or clears.  Of the 96
    showers of 10 GeV 41 at a time are in flight: the next are admitted by the
    counts of live tracks in the scratch array."""
    jobs = []
    for wl, kw in ((_large(96, 10_000.0), dict()), (_small(200), dict(block_size=64))):
        ctx = gvmod.Context(wl, gvmod.gv_default_config(stack_capacity=1 << 16, **kw))
        alone, calls = [], []
        _static_calls(gvmod, ctx, wl, 1, alone)
        jobs.append((ctx, wl, alone[0], calls))
    threads = [threading.Thread(target=_static_calls, args=(gvmod, ctx, wl, 40, calls)) for ctx, wl, _, calls in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, wl, alone, calls in jobs:
        assert alone[0] == 0 and len(calls) == 40
        for rc, counters, edep, esc in calls:
            assert rc == 0, gvmod.load().gv_strerror(rc)
            assert counters == alone[1]
            assert np.abs(edep - alone[2]).max() < 1e-9 * 1e4 and np.abs(esc - alone[3]).max() < 1e-9 * 1e4
        ctx.close()
