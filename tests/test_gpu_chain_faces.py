"""Every face of the 3D sweep, one by one, against the plain FP64 kernel's (small step budgets take it;
every face tallied there, while here x- and y-faces are tallied from shared item lists and the z-faces
follow from the cells' balance). Equal decisions: a face differs only where a particle passes
within FP32 rounding of an edge between two faces and takes the neighbouring one, so by a few particle
weights, in few places (the bounds of the 2D comparison: 4 weights; over 1 % of a weight in fewer than
2 % of the faces of any kind)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

PLAIN = {"precision": 0, "tally": 0, "schedule": 0, "step_budget": (1 << 24) - 1}
ONE = np.array([1.0])
WALL = np.array([1.0, 0.0, 0.5, 0.2, 0.0, 0.8])


def box(kind):
    rng = np.random.default_rng(7)
    if kind == "two_material":
        inst = WL.two_material_box(12)
        inst.wall_T = WALL
        return inst
    n, tau = {"ragged": ((17, 5, 9), rng.uniform(0.05, 0.6, 17 * 5 * 9)), "flat": ((24, 23, 1), rng.uniform(0.1, 1.0, 24 * 23)),
              "column": ((1, 2, 60), rng.uniform(0.1, 1.0, 120)), "uniform": ((14, 13, 12), np.full(14 * 13 * 12, 0.4))}[kind]
    return WL.Instance(3, n, (1.0, 0.8, 1.2), tau[None], WALL, rng.uniform(0, 1, int(np.prod(n))))


@pytest.mark.parametrize("opt", [{}, {"tally": 2}, {"refill_lanes": 32}], ids=str)
@pytest.mark.parametrize("kind", ["two_material", "ragged", "flat", "column", "uniform"])
def test_every_face(kind, opt):
    inst, N = box(kind), 150
    n, h = inst.n, [inst.L[a] / inst.n[a] for a in range(3)]
    V = h[0] * h[1] * h[2]
    T = np.random.default_rng(5).uniform(0.1, 1.0, inst.ncells)
    src = inst.source if inst.source is not None else np.zeros(inst.ncells)
    wmax = max(float((V * (T / inst.tau[0] + src)).max()) / N, max(V / x for x in h) * WALL.max() / 4 / N)
    a, b = [gpu_solver([inst], ONE, ONE, N, N, seed=3, **o).sweep(torch.as_tensor(T, device="cuda"), 1) for o in (opt, PLAIN)]
    assert a["counters"].tolist() == b["counters"].tolist()
    counts = [(n[0] + 1) * n[1] * n[2], n[0] * (n[1] + 1) * n[2], n[0] * n[1] * (n[2] + 1)]
    for x, y in zip(a["F"].split(counts), b["F"].split(counts)):
        d = (x - y).abs()
        assert float(d.max()) <= 4 * wmax
        assert float((d > 0.01 * wmax).double().mean()) < 0.02
        assert float(y.abs().max()) > wmax  # they carry flux (a few weights each: the second bound is the sharp one)
