"""Plans whose transform solve is not refined (precision "fp32", or "mixed" with refine_iters = 0):
their results hold the rounding of every FP32 step, so each path of a call has to take the same
steps.
"""
import pytest
import torch

from paper_2304_14690_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

UNREFINED = [("fp32", 4), ("mixed", 0)]


@pytest.fixture(scope="module")
def pc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2304_14690_gb300 import pc
    assert torch.cuda.is_available()
    return pc


@pytest.mark.parametrize("knn", [None, 10, 16])
@pytest.mark.parametrize("precision,iters", UNREFINED)
def test_batch_equals_single(pc, precision, iters, knn):
    """The batched transfer rounds the fluxes as the single call does, at every neighbour count (12 and
    27 have kernels of their own). In a small disturbance of a uniform flow the fluxes cancel, and
    their last bits reach the source of a few cells."""
    plans, args, singles = [], [], []
    for n, lo, hi in [((400, 320), "IW", "DW"), ((100, 60), "PW", "PW")]:
        q = wl.generic(dim=2, n=n, h=(1 / 64,) * 2, bc_lo=lo, bc_hi=hi, seed=81, knn=knn)
        plan = pc.Plan(q, precision=precision, refine_iters=iters)
        g = torch.Generator(device="cuda").manual_seed(1)
        u = 1.0 + 1e-5 * torch.randn(q.u_star.shape, generator=g, device="cuda", dtype=torch.float64)
        singles.append([t.clone() for t in plan.project(u)[:3]])
        p, uo, f = plan.alloc_outputs()
        plans.append(plan)
        args.append(dict(dt=q.dt, u_star=u, p=p, u=uo, f=f))
    pc.project_batch(plans, args)
    torch.cuda.synchronize()
    for a, want in zip(args, singles):
        assert all(torch.equal(x, y) for x, y in zip((a["p"], a["u"], a["f"]), want))
    for plan in plans:
        plan.close()
