"""Sample i of gv_unit_sample does not depend on how many samples its call
draws: below and from 2^20 on the table samples come from two kernels with the
same arithmetic."""
import numpy as np
import pytest

from paper_2005_00949_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1], ids=["mixed", "fp64"])
@pytest.mark.parametrize("model", range(6))
def test_samples_do_not_depend_on_the_size_of_the_call(model, prec):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2005_00949_gb300 import gv
    ctx = gv.Context(W.pbps_electrons(1), gv.gv_default_config(precision=prec, stack_capacity=1 << 12))
    n = (1 << 20) + 4321
    lo = [1e-3, 2.0, 1.5, 3.0, 2.0, 1e-3][model]  # from the lowest energies of each model's table on
    energy = torch.from_numpy(lo * 10.0 ** (8.0 * np.random.default_rng(model).random(n))).cuda()
    large = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    ctx.gv_unit_sample(model, 0, energy, 99, large)
    for m in (1, 1000, (1 << 20) - 1):
        small = torch.zeros((m, 3), dtype=torch.float64, device="cuda")
        ctx.gv_unit_sample(model, 0, energy[:m], 99, small)
        assert torch.equal(small, large[:m])
    ctx.close()
