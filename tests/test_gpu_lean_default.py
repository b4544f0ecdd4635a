"""Variant 0 of the compile-time FP32 transform passes at every length they have. A grid takes it where
an axis has no looped pass (here n = 18: M = 9 is odd) or beyond about a million cells; smaller grids
with looped passes on every axis, as in test_gpu_lean, take those or the one-launch solve, with the
same bits. Against the CPU oracle's Poisson solve, every boundary pair, rows and columns, ragged tiles.
"""
import numpy as np
import pytest
import torch

from oracle import grid as G
from oracle import poisson as P
from paper_2304_14690_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LEAN_M = [16, 32, 48, 64, 96, 128, 192, 256, 384, 512]
KINDS = {"PP": ("P", "P"), "NN": ("W", "W"), "DD": ("D", "D"), "ND": ("I", "D"), "DN": ("D", "W")}
OTHER = ["NN", "PP", "DD", "ND", "DN"]
TOL = {"fp32": 1e-5, "mixed": 1e-10}   # as in test_gpu_parity (relative L2 of p)


@pytest.fixture(scope="module")
def pc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2304_14690_gb300 import pc
    assert torch.cuda.is_available()
    return pc


def _check(pc, kinds, n, seed):
    d = len(n)
    rng = np.random.default_rng(seed)
    h = tuple(float(rng.uniform(0.5, 2.0)) / m for m in n)
    lo, hi = [KINDS[k][0] for k in kinds], [KINDS[k][1] for k in kinds]
    s = rng.normal(size=n)
    ref, _ = P.solve(s, G.Grid(d, n, (0.0,) * d, h, tuple(lo), tuple(hi)))
    for precision, tol in TOL.items():
        plan = pc.GridPlan(d, n, h, lo, hi, precision=precision)
        p = plan.solve_poisson(torch.as_tensor(s, device="cuda"))[0].cpu().numpy()
        plan.close()
        assert np.linalg.norm(p - ref) <= tol * np.linalg.norm(ref), (kinds, precision)


@pytest.mark.parametrize("M", LEAN_M)
@pytest.mark.parametrize("orient", ["col", "row"])
def test_variant0_matches_oracle(pc, M, orient):
    """Each length along axis 0 (forward, division, inverse) or axis 1 (forward, inverse)."""
    for i, kind in enumerate(KINDS):
        kinds = (kind, OTHER[i]) if orient == "col" else (OTHER[i], kind)
        _check(pc, kinds, (2 * M, 18) if orient == "col" else (18, 2 * M), 6000 + 17 * M + i)


@pytest.mark.parametrize("n", [(18, 32, 10), (18, 96, 10), (10, 256, 18), (18, 10, 384)])
def test_variant0_3d_matches_oracle(pc, n):
    """Column passes of axis 1 and rows of the last axis between axes without a looped pass."""
    for i, kinds in enumerate([("NN", "NN", "NN"), ("PP", "DD", "ND"), ("DN", "PP", "NN")]):
        _check(pc, kinds, n, 7000 + i + sum(n))


def test_variant0_batch_equals_single(pc):
    """Batched launches of variant 0 give each problem the bits of its own call."""
    plans, args, singles = [], [], []
    for i, n in enumerate([(256, 18), (18, 128), (1024, 18), (64, 18)]):
        q = wl.generic(dim=2, n=n, h=(1 / 64,) * 2, bc_lo="IW", bc_hi="DW", seed=60 + i)
        plan = pc.Plan(q, precision="mixed")
        u = torch.as_tensor(q.u_star, device="cuda")
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
