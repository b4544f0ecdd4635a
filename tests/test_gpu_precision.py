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
