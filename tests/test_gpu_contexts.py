"""Several contexts alive at once, of sizes that need different amounts of shared memory: the kernels'
limits belong to the process, and a later, smaller context must not lower them for an earlier one.
Every call of the first context gives what it gave before the others were made."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

ONE = np.array([1.0])


def inst(n, vary):
    nc, d = int(np.prod(n)), len(n)
    tau = np.random.default_rng(2).uniform(0.05, 0.5, (1, nc)) if vary else np.full((1, nc), 0.3)
    return WL.Instance(d, tuple(n) + (1,) * (3 - d), (1.0,) * 3, tau, np.linspace(0.1, 0.9, 2 * d))


def use(s, R=None):
    """Event counts and R of a sweep (atomic sums: equal to rounding), and a correction for given
    tallies (fixed order: equal to the bit)."""
    T = torch.linspace(0.1, 0.9, s.total_cells, dtype=torch.float64, device="cuda")
    out = s.sweep(T, 1)
    R = out["R"].clone() if R is None else R
    half, _ = s.macro(R)
    its = s.newton_step(T, half, R)
    return out["counters"].tolist(), out["R"], its, half, R


@pytest.mark.parametrize("opt", [{}, {"cg_rtol": 1e-8}, {"tally": 2}, {"refill_lanes": 8}], ids=str)
@pytest.mark.parametrize("big,small", [((1024, 3), (64, 3)), ((128, 128), (8, 8)), ((20000,), (8,)), ((40, 40, 20), (5, 5, 5))], ids=str)
@pytest.mark.parametrize("vary", [False, True])
def test_a_later_small_context_leaves_an_earlier_one_alone(big, small, vary, opt):
    a = gpu_solver([inst(big, vary)], ONE, ONE, 4, 4, seed=1, **opt)
    first = use(a)
    b = gpu_solver([inst(small, vary)], ONE, ONE, 4, 4, seed=1, **opt)
    use(b)
    again = use(a, first[4])
    assert again[0] == first[0] and again[2] == first[2]
    assert float((again[1] - first[1]).abs().max()) <= 1e-9 * float(first[1].abs().max())
    assert torch.equal(again[3], first[3])
