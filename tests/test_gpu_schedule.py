"""The schedule of the transform passes as callers keep it: read, written back, carried to another
plan of the same grid.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2304_14690_gb300 import pc
    assert torch.cuda.is_available()
    return pc


def _source(n):
    return torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(sum(n)), device="cuda", dtype=torch.float64)


# one cluster, one cooperative grid, 3D, beyond the one-launch solve, an axis without a looped pass (M = 9)
@pytest.mark.parametrize("n", [(64, 64), (200, 256), (48, 40, 36), (2048, 640), (18, 64)], ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_schedule_written_back(pc, precision, n):
    """Setting what was read changes nothing, and a plan set away from it comes back to the same bits."""
    d = len(n)
    plan = pc.GridPlan(d, n, (1 / 64,) * d, "WDW"[:d], "WWW"[:d], precision=precision)
    s = _source(n)
    want, slots = plan.solve_poisson(s)[0].clone(), plan.slots()
    for a in range(d):
        plan.set_slots(a, slots[a])
    assert torch.equal(plan.solve_poisson(s)[0], want)
    for a in range(d):
        plan.set_slots(a, 8)
    plan.solve_poisson(s)
    for a in range(d):
        plan.set_slots(a, slots[a])
    assert plan.slots() == slots and torch.equal(plan.solve_poisson(s)[0], want)
    plan.close()
