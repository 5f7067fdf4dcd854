"""The filtered FP64 sweep against the plain FP64 kernel (which small step budgets take), at the
edges of its emitter tiles, face segments and queues: equal event counts, and tallies that are
the same FP64 terms added in another order (n terms: n 2^-53 relative, 1e-11 for the counts
here; the faces are measured against their largest value, of which they are differences)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402
from test_gpu_land import C2, SHAPES, V2, instances  # noqa: E402

PLAIN = {"step_budget": (1 << 24) - 1}


def compare(ins, C, v, particles, T0, **kw):
    got = []
    for opt in ({}, PLAIN):
        s = gpu_solver(ins, C, v, particles, particles, seed=21, precision=0, tally=0, schedule=0, **opt)
        T = torch.as_tensor(T0, device="cuda")
        got.append(s.sweep(T, 2, **kw))
    a, b = got
    assert a["counters"].tolist() == b["counters"].tolist()
    for key in ("R", "W", "F", "wall"):
        if b[key] is None:
            assert a[key] is None
            continue
        scale = float(b[key].abs().max())
        assert scale > 0 and float((a[key] - b[key]).abs().max()) <= 1e-11 * scale, key


@pytest.mark.parametrize("particles", [2, 17, 700])
@pytest.mark.parametrize("shape", SHAPES)
def test_filtered_sweep_equals_the_plain_kernel(shape, particles):
    ins = instances(shape)
    T = np.random.default_rng(4).uniform(0.0, 1.0, sum(i.ncells for i in ins))
    T[::7] = 0.0
    compare(ins, C2, V2, particles, T)


@pytest.mark.parametrize("want", [{"want_W": False}, {"want_F": False}, {"want_F": False, "want_wall": False}])
def test_outputs_left_out(want):
    ins = instances("chains_2d")
    compare(ins, C2, V2, 50, np.ones(sum(i.ncells for i in ins)), **want)


def test_more_open_faces_than_the_queue_holds():
    # flights of hundreds of cells: the bound of a row grows with its distance, and the faces
    # left open exceed one in eight particles
    n = (700, 600)
    inst = WL.Instance(2, n, (1.0, 1.0), np.full((1, n[0] * n[1]), 5.0), np.array([1.0, 0.0, 0.5, 0.0]))
    compare([inst], np.array([1.0]), np.array([1.0]), 4, np.full(inst.ncells, 0.4))


def test_heated_segment_and_long_film():
    wl = WL.hot_segment_rectangle(Kn=0.3, nx=37, ny=21, particles=40)
    compare(wl.instances, wl.C, wl.v, 40, np.linspace(0.1, 0.9, 37 * 21))
    wl = WL.multiscale_slab(2500, 30)
    compare(wl.instances, wl.C, wl.v, 30, np.linspace(0.1, 0.9, 2500))
