"""The correction solve at the edges of its teams of blocks, strips, chunks and levels: the residual
of the solution under the FP64 operator meets the tolerance asked for. With T = T_half = 0 the
step returns theta dT, so dT is known to rounding (condition number x 2^-53: below 1e-9 here)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver, oracle_problem  # noqa: E402

ONE = np.array([1.0])


def uniform(n, tau=0.3):
    return WL.Instance(len(n), tuple(n) + (1,) * (3 - len(n)), (1.0,) * 3, np.full((1, int(np.prod(n))), tau),
                       np.linspace(0.1, 0.9, 2 * len(n)))


def mixed(n, seed=3):
    rng = np.random.default_rng(seed)
    i = uniform(n)
    i.tau[:] = rng.uniform(0.05, 0.5, i.tau.shape)
    return i


def check(ins, rtol):
    from oracle import oracle as O
    s = gpu_solver(ins, ONE, ONE, 4, 4, seed=1, cg_rtol=rtol, cg_maxit=20000)
    nc = sum(i.ncells for i in ins)
    R = np.random.default_rng(8).uniform(-1.0, 1.0, nc)
    out = torch.zeros(nc, dtype=torch.float64, device="cuda")
    Rd = torch.as_tensor(R, device="cuda")
    zero = torch.zeros_like(out)
    for rep in range(2):  # the barriers are as the first call left them
        out.zero_()
        its = s.newton_step(zero, out, Rd)
        assert its >= 1
    off = 0
    for i in ins:
        p = oracle_problem(i, ONE, ONE, 4, 4)
        dT = out[off:off + i.ncells].cpu().numpy() / O.newton_theta(p)
        d = len(i.n) if not hasattr(i, "dim") else i.dim
        V = float(np.prod([i.L[a] / i.n[a] for a in range(d)]))
        rhs = R[off:off + i.ncells] / V
        res = rhs - O.diffusion_apply(p, dT)
        assert np.linalg.norm(res) <= (1.001 * rtol + 1e-9) * np.linalg.norm(rhs), i.n
        off += i.ncells


@pytest.mark.parametrize("rtol", [1e-3, 1e-8])
@pytest.mark.parametrize("n", [(1,), (2,), (129,), (1024,), (1, 5), (128, 128), (129, 3), (3, 131), (64, 200), (260, 257)])
def test_separable(n, rtol):
    check([uniform(n)], rtol)


@pytest.mark.parametrize("rtol", [1e-3, 1e-8])
@pytest.mark.parametrize("n", [(3, 2, 1), (16, 16, 16), (17, 16, 16), (33, 20, 18), (90, 70), (5000,)])
def test_multigrid(n, rtol):
    check([mixed(n)], rtol)


@pytest.mark.parametrize("rtol", [1e-3, 1e-8])
def test_both_kinds_and_uneven_sizes(rtol):
    check([uniform((60, 60)), mixed((20, 90)), uniform((7, 5)), mixed((64, 64)), mixed((3, 3))], rtol)


def test_more_instances_than_blocks():
    check([uniform((9, 6 + k % 5)) for k in range(200)] + [mixed((8, 5 + k % 7)) for k in range(200)], 1e-3)
