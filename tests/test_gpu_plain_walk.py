"""Comparisons with the plain FP64 kernels (one thread per particle, cell by cell; step budgets below
2^24 select them), which share no decision with the fast paths: with the default budget FP64 tracking
filters its decisions in FP32 by the same positions and bounds as the landing sweeps, so that a
comparison with it would not show a bound that is too small. Every plain context must have replayed
nothing. Tolerances are those of the comparisons with FP64 tracking in the tests they come from."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_configs as configs  # noqa: E402
import test_gpu_fp32_exact as exact  # noqa: E402
import test_gpu_parity as parity  # noqa: E402
import test_gpu_variable_tau as variable  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402
from paper_2506_09465_gb300 import workloads as WL  # noqa: E402

PLAIN = {"precision": 0, "tally": 0, "schedule": 0, "step_budget": (1 << 24) - 1}


@pytest.fixture
def plain(monkeypatch):
    """FP64 contexts of the tests' modules on the plain kernels; checked at the end."""
    made = []

    def make(*args, **opt):
        if opt.get("precision") != 0:
            return gpu_solver(*args, **opt)
        made.append(gpu_solver(*args, **{**opt, **PLAIN}))
        return made[-1]

    for module in (configs, exact, parity, variable):
        monkeypatch.setattr(module, "gpu_solver", make)
    yield made
    assert made and all(s.replayed() == 0 for s in made)


@pytest.fixture(scope="module")
def cavity_pair():
    # the benchmark batch (128^2, four Knudsen numbers, 1024 particles per cell and wall face)
    wl = WL.cavity_sweep(128, exact.KNS, 1024)
    fast = gpu_solver(wl.instances, [1.0], [1.0], 1024, 1024, seed=0)
    return wl, fast, [gpu_solver(i, [1.0], [1.0], 1024, 1024, seed=0, instance_base=j, use_graphs=0, **PLAIN)
                      for j, i in enumerate(wl.instances)]


def test_bench_cavity_sweep(cavity_pair):
    exact.test_bench_cavity_sweep_equals_fp64_walk(cavity_pair)
    assert all(s.replayed() == 0 for s in cavity_pair[2])


def test_bench_cavity_steady_state(cavity_pair):
    exact.test_bench_cavity_steady_state_equals_fp64_walk(cavity_pair)
    assert all(s.replayed() == 0 for s in cavity_pair[2])


@pytest.mark.parametrize("n", [96, 180])
def test_two_group_faces(plain, n):
    parity.test_two_group_face_tallies_match_plain_fp64_faces(n)


def test_box_batch(plain, orc):
    configs.test_box_batch_conserves_and_matches_standalone(orc)


@pytest.mark.parametrize("case", list(variable.CASES))
def test_variable_tau_steady(plain, orc, case):
    variable.test_variable_tau_steady_matches_oracle(orc, case)


@pytest.mark.parametrize("kind", ["square", "nongray", "box"])
def test_steady_state_of_fp64_tracking(kind):
    # The filtered FP64 walk's steady loop and adjoint (landing sweeps) against the plain kernels': the
    # solutions of the same frozen map to the iteration's tolerance, 1e-9 of the 2-norm on either side
    # with steps that shrink by half or more; the largest value is at least the norm over the
    # square root of the cells (512 at most): 2 x 1e-9 x 23
    if kind == "square":
        inst, C, v = WL.random_instance(np.random.default_rng(4), 2, (24, 18), 1, (0.02, 1.0), source=True), [1.0], [1.0]
    elif kind == "nongray":
        wl = WL.nongray_square(20, 4, 64)
        inst, C, v = wl.instances[0], wl.C, wl.v
    else:
        inst, C, v = WL.two_material_box(8), [1.0], [1.0]
    g = torch.linspace(0.1, 1.0, inst.ncells, dtype=torch.float64, device="cuda")
    got = []
    for opt in ({"precision": 0, "tally": 0, "schedule": 0}, PLAIN):
        s = gpu_solver([inst], C, v, 64, 64, seed=3, cg_rtol=1e-10, cg_maxit=20000, **opt)
        T, _, _ = s.solve_steady(None, 1e-9, 400)
        got.append((T, *s.adjoint(g, 1e-9, 400)))
    for a, b in zip(*got):
        assert float((a - b).abs().max()) <= 4.6e-8 * float(b.abs().max())
