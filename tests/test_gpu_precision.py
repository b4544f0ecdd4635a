"""What FP64 and correctly rounded FP32 steps of the solve owe their callers: the division by the
eigenvalues and the mean of the source.
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


@pytest.mark.parametrize("n,lo,hi", [((100, 200), "IW", "DW"), ((400, 60), "PD", "PW"), ((20, 24, 40), "DWW", "DWD")],
                         ids=["100x200", "400x60", "20x24x40"])
def test_division_by_large_eigenvalues(pc, n, lo, hi):
    """Eigenvalue sums up to 2.5e38, beyond 2^126, where the approximate division returns zero: lengths
    without a compile-time pass divide with IEEE rounding, and the refined solve agrees with the
    FP64 one to the refinement's tolerance (1e-10, as in test_gpu_parity)."""
    d = len(n)
    h = (4.0 * d / 2.5e38) ** 0.5   # the largest sum is 4 d / h^2
    s = 1e20 * _source(n)
    p = {}
    for precision in ("mixed", "fp64"):
        plan = pc.GridPlan(d, n, (h,) * d, lo, hi, precision=precision)
        p[precision] = plan.solve_poisson(s)[0].clone()
        plan.close()
    assert float((p["mixed"] - p["fp64"]).norm() / p["fp64"].norm()) <= 1e-10


def test_mean_of_the_source_in_64_bits(pc):
    """The mean of 1 + r and 1 - r in rows of four, r = 2^-24 + 15 * 2^-51, on 64 x 64 cells. A thread of
    the sum takes cells 256 apart, two of each: in FP64 its sums are exact (r is a multiple of 2^-51,
    and 3 + r has 53 bits), and all that follow add fours. As FP32 pairs both values lose their last
    bits, in the same direction."""
    r = 2.0 ** -24 + 15 * 2.0 ** -51
    s = torch.ones((64, 64), dtype=torch.float64, device="cuda")
    up = (torch.arange(64, device="cuda") // 4) % 2 == 0
    s[up] += r
    s[~up] -= r
    plan = pc.GridPlan(2, (64, 64), (1 / 64, 1 / 64), "WW", "WW", precision="mixed")
    assert plan.solve_poisson(s, stats=True)[1]["removed_mean"] == 1.0
    plan.close()
