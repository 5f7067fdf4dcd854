"""The 3D sweep's three phases (emit, walk, end) at the edges of their lists: equal event counts and
real collisions with the plain FP64 kernel (which small step budgets take). Every decision is the
FP64 walk's, so R differs by the order of its FP64 terms only (1e-11); a null candidate within
rounding of a face may be counted in the neighbouring cell of W, so W is compared by its sum, and
a face crossed within rounding of an edge may take the neighbouring face, so F by the walls' power
(1e-6 of the largest)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

C2, V2 = np.array([0.7, 0.3]), np.array([1.0, 2.5])


def boxes(kind):
    rng = np.random.default_rng(11)
    wall = np.array([1.0, 0.0, 0.5, 0.2, 0.0, 0.8])

    def inst(n, tau):
        return WL.Instance(3, n, (1.0, 0.8, 1.2), tau, wall, rng.uniform(0, 1, int(np.prod(n))))

    if kind == "one_cell":
        return [inst((1, 1, 1), np.full((2, 1), 0.3))]
    if kind == "all_real":
        return [inst((7, 3, 5), np.full((2, 105), 0.2))]
    if kind == "thin":
        return [inst((33, 1, 4), rng.uniform(0.02, 1.0, (2, 132)))]
    if kind == "chains":  # a hundred null candidates per flight, several per cell
        tau = np.full((2, 9 * 8 * 7), 3.0)
        tau[:, ::97] = 0.01
        return [inst((9, 8, 7), tau)]
    return [inst((4, 4, 4), rng.uniform(0.01, 2.0, (2, 64))), inst((1, 2, 3), np.full((2, 6), 5.0)),
            inst((12, 5, 9), rng.uniform(0.05, 0.1, (2, 540)))]


@pytest.mark.parametrize("opt", [{}, {"refill_lanes": 32}, {"refill_lanes": 1, "warp_grab": 33}, {"tally": 2}])
@pytest.mark.parametrize("particles", [2, 37])
@pytest.mark.parametrize("kind", ["one_cell", "all_real", "thin", "chains", "batch"])
def test_equals_the_plain_kernel(kind, particles, opt):
    ins = boxes(kind)
    T0 = np.random.default_rng(5).uniform(0.1, 1.0, sum(i.ncells for i in ins))
    T0[::5] = 0.0
    got = []
    for o in (opt, {"precision": 0, "tally": 0, "schedule": 0, "step_budget": (1 << 24) - 1}):
        s = gpu_solver(ins, C2, V2, particles, particles, seed=3, **o)
        got.append(s.sweep(torch.as_tensor(T0, device="cuda"), 2))
    a, b = got
    assert a["counters"].tolist() == b["counters"].tolist()
    scale = float(b["R"].abs().max())
    assert float((a["R"] - b["R"]).abs().max()) <= 1e-11 * scale
    assert abs(float(a["W"].sum() - b["W"].sum())) <= 1e-10 * float(b["W"].sum().abs())
    assert float((a["wall"] - b["wall"]).abs().max()) <= 1e-6 * float(b["wall"].abs().max())


def test_outputs_left_out():
    ins = boxes("batch")
    T = torch.ones(sum(i.ncells for i in ins), dtype=torch.float64, device="cuda")
    s = gpu_solver(ins, C2, V2, 50, 50, seed=3)
    full = s.sweep(T, 1)
    for want in ({"want_W": False}, {"want_F": False, "want_wall": False}):
        part = s.sweep(T, 1, **want)
        assert part["counters"].tolist() == full["counters"].tolist()
        assert float((part["R"] - full["R"]).abs().max()) <= 1e-11 * float(full["R"].abs().max())
