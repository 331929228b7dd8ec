"""The end of a transport: the generation that finds nothing left to plan.
With dependent launch its successor's blocks already run, so a block may look
at the done flag while it is being set; whatever it sees, all of its threads
must see it."""
import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(generations_per_graph=2), dict(generations_per_graph=64, device_loop=0),
                                dict(precision=1), dict(process_sort=0), dict(block_size=64)],
                         ids=["default", "short-body", "host-loop", "fp64", "no-sort", "64"])
def test_many_short_transports_end_alike(kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    wl = W.photon_slab(3, 1.0)
    ctx = gv.Context(wl, gv.gv_default_config(per_event_counts=1, stack_capacity=1 << 12, **kw))
    first = ctx.transport(per_event=True)
    assert first["status"] == 0 and first["counters"]["generations"] >= 1
    edep = np.zeros((3, ctx.n_subtotal))
    counts = np.zeros((3, gv.NCOUNT), dtype=np.int64)
    for _ in range(500):
        r = ctx.gv_transport(wl.primaries, 3, wl.seed, edep, event_counts=counts)
        assert r.status == 0
        assert np.array_equal(counts[:, :11], first["counts"][:, :11])
        assert np.array_equal(edep, first["edep"])
    ctx.close()
