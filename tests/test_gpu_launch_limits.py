"""What contexts and threads share: the limit of a kernel's dynamic shared
memory.  A context made later, or a call on another thread, that needs less of
it must leave room for those that need more."""
import dataclasses
import threading

import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gvmod():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    return gv


def _large(n=60):
    """Four materials and 800 sub-slabs."""
    return dataclasses.replace(W.pbps_electrons(n, 300.0), n_layers=100,
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
