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


# lengths with a compile-time pass (64, 256), without one (100, 200, 400, 40, 60), and both
SOLVES = [((100, 200), "WP", "WP"), ((400, 400), "PP", "PP"), ((64, 200), "ID", "DW"), ((64, 256), "WW", "WW"),
          ((40, 60, 100), "WPD", "WPW")]


@pytest.mark.parametrize("n,lo,hi", SOLVES, ids=["x".join(map(str, s[0])) for s in SOLVES])
def test_mixed_without_sweeps_is_the_fp32_solve(pc, n, lo, hi):
    """A mixed plan without sweeps returns the bits of an FP32 plan: one solve and one projection."""
    s = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(sum(n)), device="cuda", dtype=torch.float64)
    q = wl.generic(dim=len(n), n=n, h=(1 / 64,) * len(n), bc_lo=lo, bc_hi=hi, seed=3)
    u = torch.as_tensor(q.u_star, device="cuda")
    got = []
    for precision, iters in UNREFINED:
        grid = pc.GridPlan(len(n), n, (1 / 64,) * len(n), lo, hi, precision=precision, refine_iters=iters)
        plan = pc.Plan(q, precision=precision, refine_iters=iters)
        got.append([grid.solve_poisson(s)[0].clone()] + [t.clone() for t in plan.project(u)[:3]])
        grid.close()
        plan.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))
