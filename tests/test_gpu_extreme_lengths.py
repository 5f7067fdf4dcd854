"""Mean free paths and cells beyond FP32's range: every call takes them, and the results are the plain
FP64 kernel's (which small step budgets take). The FP64 terms are added in another order: 1e-11."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

PLAIN = {"precision": 0, "tally": 0, "schedule": 0, "step_budget": (1 << 24) - 1}
FP64 = {"precision": 0, "tally": 0, "schedule": 0}
C2, V2 = np.array([0.6, 0.4]), np.array([1.0, 0.5])


def instance(n, tau, h=1.0):
    d, nc = len(n), int(np.prod(n))
    return WL.Instance(d, tuple(n) + (1,) * (3 - d), (h * 1.0, h * 0.7, h * 1.2)[:d] + (1.0,) * (3 - d),
                       np.array([[tau], [0.2 * h]]) * np.ones((2, nc)), np.linspace(0.1, 0.9, 2 * d))


def close(a, b, tol=1e-11):
    assert float((a - b).abs().max()) <= tol * float(b.abs().max())


GRIDS = [(40,), (9, 13), (5, 4, 6)]


@pytest.mark.parametrize("opt", [FP64, {}, {"tally": 2}], ids=["fp64", "fp32", "fp32_k32"])
@pytest.mark.parametrize("n,tau", [((9, 13), 1e37), ((9, 13), 1e39), ((5, 4, 6), 1e37), ((5, 4, 6), 1e39),
                                   ((1,), 1e37), ((1,), 1e300), ((1, 1), 1e300), ((1, 1, 1), 1e300)], ids=str)
def test_endless_free_paths(n, tau, opt):
    # v tau_maj infinite in FP32 for one of the two bands (nearly so at 1e37: some paths are). On other
    # grids the correction's operator is singular in FP64 at such tau and no context is made.
    inst = instance(n, tau)
    got = []
    for o in (opt, PLAIN):
        s = gpu_solver([inst], C2, V2, 20, 20, seed=5, newton=0, use_graphs=0, **o)
        T = torch.linspace(0.2, 0.9, inst.ncells, dtype=torch.float64, device="cuda")
        sweep = s.sweep(T, 0)
        steady, _, _ = s.solve_steady(T, 0.0, 1, raise_on_noconv=False)
        adjoint = s.adjoint(torch.linspace(0.1, 1.0, inst.ncells, dtype=torch.float64, device="cuda"), 1e6)
        got.append((sweep, steady, adjoint))
    (a, sa, aa), (b, sb, ab) = got
    assert a["counters"].tolist() == b["counters"].tolist()
    tol = 1e-9 if opt.get("tally") == 2 else 1e-11
    close(a["R"], b["R"], tol)
    close(sa, sb, tol)
    for x, y in zip(aa, ab):
        close(x, y)


@pytest.mark.parametrize("h", [1e39, 1e-39])
@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_cells_beyond_fp32(n, h):
    # FP64 tracking: the units are the caller's
    inst = instance(n, 0.3 * h, h)
    got = []
    for o in (FP64, PLAIN):
        s = gpu_solver([inst], C2, V2, 20, 20, seed=5, newton=0, use_graphs=0, **o)
        got.append(s.sweep(torch.linspace(0.2, 0.9, inst.ncells, dtype=torch.float64, device="cuda"), 0))
    a, b = got
    assert a["counters"].tolist() == b["counters"].tolist()
    close(a["R"], b["R"])
