"""Waits inside the one-launch solves that run out: the call or the next one says so, the whole result
is NaN, and the plan works again. The limit is an argument, so a limit of one poll makes the waits
give up at once; the kernels then end by themselves.

On the 96 x 1000 grid the row passes have 96 tiles and the column passes 125, so 29 thread blocks
arrive at the first wait while the others still transform their rows: they give up there, and with
them gone every other block gives up at the second wait.
"""
import pytest
import torch

from paper_2304_14690_gb300 import workloads as wl

N, H = (96, 1000), (1 / 96, 1 / 96)


@pytest.fixture(scope="module")
def pc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2304_14690_gb300 import pc
    return pc


def test_limit_needs_a_plan(pc):
    assert pc.load().pc_plan_set_wait_limit(None, 0) == 1


def _timeout(pc, call):
    with pytest.raises(pc.PcError) as e:
        call()
    assert e.value.status == 8   # PC_ERR_TIMEOUT


def _source():
    return torch.randn(N, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda", dtype=torch.float64)


@pytest.mark.gpu
@pytest.mark.parametrize("bc", ["ID", "WW"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("graphs", [True, False])
def test_solve_that_gave_up(pc, precision, bc, graphs):
    plan = pc.GridPlan(2, N, H, bc[0] + "W", bc[1] + "W", precision=precision)
    plan.graphs(graphs)
    s = _source()
    want = plan.solve_poisson(s)[0].clone()
    plan.set_wait_limit(1)
    p = plan.solve_poisson(s)[0]
    torch.cuda.synchronize()
    assert bool(torch.isnan(p).all())
    _timeout(pc, lambda: plan.solve_poisson(s))                  # device arrays: the next call says so
    _timeout(pc, lambda: plan.solve_poisson(s.cpu()))            # host arrays: the call itself
    if precision == "fp64":
        _timeout(pc, lambda: plan.solve_poisson(s, stats=True))  # (mixed statistics take launches)
    plan.set_wait_limit(1 << 22)
    assert torch.equal(plan.solve_poisson(s)[0], want)
    plan.close()


@pytest.mark.gpu
def test_other_calls_report_it(pc):
    """The projection, the force iteration, the batch and the autotuner."""
    q = wl.generic(dim=2, n=N, h=H, bc_lo="IW", bc_hi="DW", obstacles=[("circle", (0.5, 5.0), 0.1)], seed=4)
    plan, other = pc.Plan(q, precision="mixed"), pc.Plan(q, precision="mixed")
    u = torch.as_tensor(q.u_star, device="cuda")
    want = [t.clone() for t in plan.project(u)[:3]]
    plan.set_wait_limit(1)
    got = plan.project(u)
    torch.cuda.synchronize()
    assert all(bool(torch.isnan(t).any()) for t in got[:2])
    outs = [p.alloc_outputs() for p in (plan, other)]
    args = [dict(dt=q.dt, u_star=u, p=o[0], u=o[1], f=o[2]) for o in outs]
    _timeout(pc, lambda: pc.project_batch([plan, other], args))
    _timeout(pc, lambda: plan.project_ib(u, max_iters=3))
    _timeout(pc, plan.autotune)
    _timeout(pc, lambda: plan.project(u, out=tuple(t.cpu() for t in outs[0])))
    plan.set_wait_limit(1 << 22)
    for a in (0, 1):
        plan.set_slots(a, 0)
    assert all(torch.equal(a, b) for a, b in zip(plan.project(u)[:3], want))
    plan.close()
    other.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_periodic_vertex_grid(pc, precision):
    """A vertex grid of periodic axes has the cell grid's transforms, and its waits."""
    plan = pc.GridPlan(2, N, H, "PP", "PP", grid_type="vertices", precision=precision)
    s = _source()
    want = plan.solve_poisson(s)[0].clone()
    plan.set_wait_limit(1)
    _timeout(pc, lambda: plan.solve_poisson(s.cpu()))
    plan.set_wait_limit(1 << 22)
    assert torch.equal(plan.solve_poisson(s)[0], want)
    plan.close()


@pytest.mark.gpu
def test_more_plans_than_pooled_words(pc):
    """Each plan reports its own waits, also those beyond the 1024 whose words share a page."""
    small = [pc.GridPlan(2, (8, 8), (1 / 8, 1 / 8), "WW", "WW") for _ in range(1023)]
    plans = [pc.GridPlan(2, N, H, "IW", "DW") for _ in range(3)]
    s = _source()
    want = plans[0].solve_poisson(s)[0].clone()
    for plan in (plans[0], plans[2]):
        plan.set_wait_limit(1)
        plan.solve_poisson(s)
    torch.cuda.synchronize()
    _timeout(pc, lambda: plans[0].solve_poisson(s))
    assert torch.equal(plans[1].solve_poisson(s)[0], want)
    _timeout(pc, lambda: plans[2].solve_poisson(s))
    for plan in small + plans:
        plan.close()
    plan = pc.GridPlan(2, N, H, "IW", "DW")
    assert torch.equal(plan.solve_poisson(s)[0], want)
    plan.close()


# one cluster and cooperative grids in 2D and 3D, both gauges
@pytest.mark.gpu
@pytest.mark.parametrize("n,lo,hi,gauge", [((64, 64), "WP", "WP", 0), ((48, 64), "ID", "WD", 0), ((64, 60), "WW", "WW", 1),
                                           ((12, 16, 20), "WWW", "WWW", 0), (N, "WW", "WW", 0), ((400, 200), "PP", "PP", 1),
                                           ((48, 40, 60), "WPW", "WPW", 0), ((64, 48, 32), "DPW", "WPD", 0),
                                           # many short lines, tiles wider than the lines side by side
                                           ((2048, 16), "IW", "DW", 0), ((16, 2048), "WD", "WW", 0), ((1200, 20), "PW", "PW", 0),
                                           ((400, 12, 12), "WWP", "WWP", 0), ((12, 200, 12), "DIP", "WDP", 0),
                                           ((32, 32, 32), "WWW", "WWW", 0)])
def test_without_waits(pc, n, lo, hi, gauge):
    """Limit 0: one launch per pass. Mixed solves keep their bits, and FP64 ones without a zero mode;
    with one, the gauge constant of the launches is summed as FP32 pairs (each thread's sum cut to
    2^-46, then eight levels of pair sums): within 2^-43 of the largest pressure."""
    d = len(n)
    s = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(sum(n)), device="cuda", dtype=torch.float64)
    zero_mode = all(a in "WIP" and b in "WIP" for a, b in zip(lo, hi))
    for precision in ("mixed", "fp64"):
        plan = pc.GridPlan(d, n, (1 / 64,) * d, lo, hi, precision=precision, gauge=gauge)
        one = plan.solve_poisson(s)[0].clone()
        plan.set_wait_limit(0)
        launches = plan.solve_poisson(s)[0]
        if precision == "mixed" or not zero_mode or gauge == 1:
            assert torch.equal(one, launches), precision
        else:
            assert float((one - launches).abs().max()) <= 2.0 ** -43 * float(one.abs().max())
        plan.close()
