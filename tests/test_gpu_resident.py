"""GPU parity of the cooperative solve (one kernel for all passes and sweeps of a grid) and of the
looped transform passes (lengths without a compile-time pass, FP64), through the C ABI.

The cases sit at the edges of their ranges: the shortest axes (M = 6), factors of 5 and 25, one
line per tile and several tiles per CTA, ragged tiles, periodic rows whose neighbours belong to
other CTAs, 3D halos on both outer axes, the largest grids of the cooperative solve and grids just
beyond it. References: the CPU oracle (relative L2 of p: FP64 1e-12, mixed 1e-10, the tolerances of
test_gpu_parity), and bit for bit the same solve with statistics, which takes one launch per pass.
"""
import numpy as np
import pytest

from oracle import grid as G
from oracle import poisson as P
from paper_2304_14690_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

KINDS = {"PP": ("P", "P"), "NN": ("W", "W"), "DD": ("D", "D"), "ND": ("I", "D"), "DN": ("D", "W")}
# (kinds, cells): every family along rows and columns, lengths with and without a compile-time pass
CASES = [(("NN", "PP"), (12, 12)), (("ND", "NN"), (20, 24)), (("PP", "DD"), (100, 40)), (("DN", "ND"), (60, 720)),
         (("NN", "NN"), (1000, 16)), (("PP", "PP"), (400, 400)), (("DD", "NN"), (96, 500)), (("NN", "ND"), (256, 2048)),
         (("ND", "NN"), (1024, 1024)), (("NN", "PP"), (1200, 900)),
         (("NN", "NN", "NN"), (12, 20, 24)), (("PP", "DN", "ND"), (36, 40, 60)), (("DD", "PP", "PP"), (64, 48, 32)),
         (("NN", "NN", "PP"), (96, 100, 80))]


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2304_14690_gb300 import pc
    assert torch.cuda.is_available()
    return pc, torch, torch.device("cuda", 0)


@pytest.mark.parametrize("kinds,n", CASES, ids=["x".join(map(str, n)) + "-" + "-".join(k) for k, n in CASES])
def test_solve_matches_oracle_and_launches(env, kinds, n):
    pc, torch, dev = env
    dim = len(n)
    rng = np.random.default_rng(7000 + sum(n))
    h = tuple(rng.uniform(0.5, 2.0) / max(n) for _ in n)
    lo, hi = [KINDS[k][0] for k in kinds], [KINDS[k][1] for k in kinds]
    s = rng.normal(size=n)
    ref, _ = P.solve(s, G.Grid(dim, n, (0.0,) * dim, h, tuple(lo), tuple(hi)))
    sd = torch.as_tensor(s, device=dev)
    for precision, tol in (("mixed", 1e-10), ("fp64", 1e-12)):
        plan = pc.GridPlan(dim, n, h, lo, hi, precision=precision)
        p, _ = plan.solve_poisson(sd)
        again, _ = plan.solve_poisson(sd)
        launches, _ = plan.solve_poisson(sd, stats=True)
        torch.cuda.synchronize()
        assert rel(p.cpu().numpy(), ref) <= tol, precision
        assert torch.equal(p, again) and torch.equal(p, launches), precision
        plan.close()


@pytest.mark.parametrize("precision", ["mixed", "fp32"])
def test_batch_equals_single_at_other_lengths(env, precision):
    """Projections at lengths without a compile-time pass, single and batched, bit for bit."""
    pc, torch, dev = env
    plans, args, singles = [], [], []
    for i, (n, lo, hi) in enumerate([((100, 60), "PW", "PW"), ((40, 200), "IW", "DW"), ((64, 50), "WD", "WW"),
                                     ((24, 20, 36), "WPD", "WPW")]):
        prob = wl.generic(dim=len(n), n=n, h=(1 / 64,) * len(n), bc_lo=lo, bc_hi=hi, seed=80 + i)
        plan = pc.Plan(prob, precision=precision)
        u = torch.as_tensor(prob.u_star, device=dev)
        singles.append([t.clone() for t in plan.project(u)[:3]])
        p, uo, f = plan.alloc_outputs()
        plans.append(plan)
        args.append(dict(dt=prob.dt, u_star=u, p=p, u=uo, f=f))
    pc.project_batch(plans, args)
    torch.cuda.synchronize()
    for a, want in zip(args, singles):
        assert all(torch.equal(x, y) for x, y in zip((a["p"], a["u"], a["f"]), want))
    for plan in plans:
        plan.close()


def test_concurrent_streams(env):
    """Cooperative solves of several plans on their own streams at once give their bits alone."""
    pc, torch, dev = env
    plans, outs, alone, streams = [], [], [], [torch.cuda.Stream() for _ in range(4)]
    src = [torch.as_tensor(np.random.default_rng(90 + i).normal(size=(n, 256)), device=dev) for i, n in enumerate((200, 240, 288, 320))]
    for s in src:
        plans.append(pc.GridPlan(2, tuple(s.shape), (1 / 64, 1 / 64), "WP", "WP", precision="mixed"))
        alone.append(plans[-1].solve_poisson(s)[0].clone())
        outs.append(torch.empty_like(s))
    torch.cuda.synchronize()
    for _ in range(5):
        for plan, s, o, st in zip(plans, src, outs, streams):
            plan.solve_poisson(s, p_out=o, stream=st)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(alone, outs))
    for plan in plans:
        plan.close()
