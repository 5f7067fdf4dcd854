"""Digits of the filtered FP64 sweep where the powers of an instance span twelve decades: a wall at
10^12 beside cells at 1 in a thick medium (mean free path 0.8 cells, so nothing crosses 40 cells:
e^-50). What a face far from the hot wall carries, and what any wall absorbs, comes from the cells
within reach alone. With n terms of sum S two orders of addition differ by at most n 2^-53 S: here
n <= reach x particles x 2 and S <= 2 x reach x the power of a cell, times the cells across. Compared with the
plain FP64 kernel (which small step budgets take). A NaN or infinite temperature must reach the
outputs that its particles touch, and no others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

PLAIN = {"step_budget": (1 << 24) - 1}
ONE = np.array([1.0])
REACH, PARTICLES = 40, 60


def instance(n, hot):
    d = len(n)
    h = 0.01
    wall = np.zeros(2 * d)
    wall[0] = hot
    return WL.Instance(d, tuple(n) + (1,) * (3 - d), tuple(h * x for x in n) + (1.0,) * (3 - d), np.full((1, int(np.prod(n))), 0.8 * h), wall)


def sweeps(inst, T, N=PARTICLES):
    out = []
    for opt in ({}, PLAIN):
        s = gpu_solver([inst], ONE, ONE, N, N, seed=7, precision=0, tally=0, schedule=0, **opt)
        out.append(s.sweep(torch.as_tensor(T, device="cuda"), 1))
    return out


def bound(inst):
    d, n = inst.dim, inst.n
    h = inst.L[0] / n[0]
    across = int(np.prod(n[1:d])) if d > 1 else 1
    power = h ** d / (0.8 * h)  # V C / tau T of a cell
    return REACH * PARTICLES * 2 * across * 2.0 ** -53 * 2 * REACH * across * power


@pytest.mark.parametrize("n", [(300,), (1500,), (130, 9), (130, 3, 4)], ids=str)
def test_powers_far_below_the_hot_wall(n):
    inst = instance(n, 1e12)
    T = np.ones(inst.ncells)
    a, b = sweeps(inst, T)
    assert a["counters"].tolist() == b["counters"].tolist()
    ends_a, ends_b, sides_a, sides_b = a["wall"][:2], b["wall"][:2], a["wall"][2:], b["wall"][2:]
    assert bool((ends_b > 0).all()) and float(ends_b.max()) < 1e3  # neither end wall takes from the hot one
    assert float((ends_a - ends_b).abs().max()) <= bound(inst)
    particles = PARTICLES * (inst.ncells + int(np.prod(inst.n[1:inst.dim])))
    assert bool(((sides_a - sides_b).abs() <= particles * 2.0 ** -53 * sides_b).all())  # the sides do
    if inst.dim == 1:
        far = slice(2 * REACH, None)  # nothing of the hot wall's gets there
        assert float(b["F"][far].abs().max()) < 1e3
        assert float((a["F"][far] - b["F"][far]).abs().max()) <= bound(inst)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n", [(300,), (30, 20), (9, 8, 7)], ids=str)
def test_one_cell_that_is_not_finite(n, value):
    inst = instance(n, 1.0)
    T = np.linspace(0.2, 0.8, inst.ncells)
    T[inst.ncells // 2] = value
    a, b = sweeps(inst, T, 20)
    for key in ("R", "W", "F", "wall"):
        assert torch.equal(torch.isfinite(a[key]), torch.isfinite(b[key])), key
        assert torch.equal(torch.isnan(a[key]), torch.isnan(b[key])), key
