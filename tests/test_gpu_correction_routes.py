"""The multigrid correction at the edges of its rule of launch (one cluster per instance where the
largest has 257 to 18,000 cells and all clusters run at once, teams of blocks otherwise): the residual
under the FP64 operator meets the tolerance, and an instance's solution does not depend on the others
beyond the rounding of the tolerance asked for (rtol 1e-10: two solutions of the same system within
2 x 1e-10 x the condition number, below 10^4 here)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import gpu_solver  # noqa: E402
from test_gpu_correction import ONE, check, mixed  # noqa: E402


@pytest.mark.parametrize("rtol", [1e-3, 1e-8])
@pytest.mark.parametrize("n", [(16, 16), (257,), (17, 61), (26, 26, 26), (27, 26, 26), (136, 133), (30, 30, 30)], ids=str)
def test_around_the_rule(n, rtol):
    check([mixed(n)], rtol)


@pytest.mark.parametrize("rtol", [1e-3, 1e-8])
@pytest.mark.parametrize("count", [1, 8, 14, 40])
def test_counts(count, rtol):
    check([mixed((11 + k % 4, 12, 10), 3 + k) for k in range(count)] + [mixed((5, 4, 1), 2)], rtol)


def test_alone_and_in_a_batch():
    ins = [mixed((20, 18, 9), 5), mixed((31, 32, 33), 6), mixed((300, 1, 1), 7)]
    rng = np.random.default_rng(1)
    R = [torch.as_tensor(rng.uniform(-1, 1, i.ncells), device="cuda") for i in ins]

    def solve(which):
        s = gpu_solver([ins[k] for k in which], ONE, ONE, 4, 4, cg_rtol=1e-10, cg_maxit=20000)
        out = torch.zeros(s.total_cells, dtype=torch.float64, device="cuda")
        s.newton_step(torch.zeros_like(out), out, torch.cat([R[k] for k in which]))
        return list(out.split([ins[k].ncells for k in which]))

    for a, b in zip(solve([0, 1, 2]), [solve([k])[0] for k in range(3)]):
        assert float((a - b).norm()) <= 2e-6 * float(b.norm())
