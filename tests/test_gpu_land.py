"""Landing sweeps (the steady loop's sweep, of which only the real collisions are read, and the
adjoint re-trace) against the full sweep and the plain FP64 re-trace of the same particles, at
the edges of their emitter tiles and task runs. Both sides add the same FP64 terms in another
order: n terms of one sign differ by at most n 2^-53 relative, 1e-11 for the counts here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402

C2, V2 = np.array([0.6, 0.4]), np.array([1.0, 0.5])


def instances(shape):
    rng = np.random.default_rng(11)
    if shape == "uniform_1d":  # 50 emitters in two tiles of 25, walls of one emitter
        return [WL.Instance(1, (50,), (1.0,), np.array([[0.3], [0.05]]) * np.ones((2, 50)), np.array([1.0, -1.0]))]
    if shape == "uniform_2d":  # narrow, ragged and single-cell grids in one batch, long flights
        return [WL.Instance(2, n, (1.0, 0.7), np.array([[t], [0.3 * t]]) * np.ones((2, n[0] * n[1])),
                            np.array([1.0, 0.0, 0.4, 0.2])) for n, t in (((5, 3), 2.0), ((33, 31), 0.02), ((1, 1), 0.5))]
    if shape == "wide_2d":  # walls far from the emitters: their coordinates round by more than the bound
        return [WL.Instance(2, (128, 96), (1.0, 0.7), np.array([[1.0], [0.7]]) * np.ones((2, 128 * 96)),
                            np.array([1.0, 0.0, 0.4, 0.2]))]
    if shape == "uniform_3d":
        return [WL.Instance(3, (7, 4, 9), (1.0, 0.5, 1.2), np.full((2, 252), 0.2), np.array([0.5, 0, 0, 1.0, 0, 0.3]))]
    dim, n = {"chains_1d": (1, (41,)), "chains_2d": (2, (13, 22)), "chains_3d": (3, (6, 9, 5))}[shape]
    inst = WL.random_instance(rng, dim, n, 2, (0.02, 1.5), source=True)
    inst.tau[1] = 0.1  # one band whose every candidate is real beside one with chains
    return [inst]


SHAPES = ["uniform_1d", "uniform_2d", "wide_2d", "uniform_3d", "chains_1d", "chains_2d", "chains_3d"]


@pytest.mark.parametrize("tally", [1, 2])
@pytest.mark.parametrize("particles", [3, 700])
@pytest.mark.parametrize("shape", SHAPES)
def test_steady_loop_sweep_equals_the_full_sweep(shape, particles, tally):
    ins = instances(shape)
    s = gpu_solver(ins, C2, V2, particles, particles, seed=9, tally=tally, newton=0, use_graphs=0)
    T = torch.as_tensor(np.random.default_rng(1).uniform(0.0, 1.0, s.total_cells), device="cuda")
    T[::7] = 0.0  # emitters without weight
    for k in range(len(ins)):
        if ins[k].source is not None:
            ins[k].source[::5] = 0.0
    want, _ = s.macro(s.sweep(T, 0)["R"])
    got, it, _ = s.solve_steady(T, 0.0, 1, raise_on_noconv=False)
    assert it == 1
    tol = 1e-11 if tally == 1 else 1e-9  # compensated FP32: about n 2^-48
    assert float((got - want).abs().max()) <= tol * float(want.abs().max())


@pytest.mark.parametrize("shape", SHAPES)
def test_adjoint_retrace_equals_the_plain_fp64_one(shape):
    ins = instances(shape)
    out = []
    for opt in ({}, {"precision": 0, "tally": 0}, {"precision": 0, "tally": 0, "step_budget": (1 << 24) - 1}):
        s = gpu_solver(ins, C2, V2, 300, 300, seed=9, newton=0, **opt)
        g = torch.as_tensor(np.random.default_rng(2).uniform(0.0, 1.0, s.total_cells), device="cuda")
        out.append(s.adjoint(g, 1e-9, 50000))  # no correction: thousands of iterations where cells are thick
    for got in out[:2]:  # FP32 and FP64 tracking; budgets below 2^24 take the plain kernel
        for a, b in zip(got, out[2]):
            assert float((a - b).abs().max()) <= 1e-11 * float(b.abs().max())
