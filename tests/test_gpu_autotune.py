"""Autotuning leaves alone the options that the context's sweep does not read: walk_k in 3D and with the
pass-synchronous schedule."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402


@pytest.mark.parametrize("kind", ["box", "square", "varying_square"])
def test_walk_k_is_searched_only_where_it_is_read(kind):
    if kind == "box":
        inst = WL.two_material_box(12)
    elif kind == "square":
        inst = WL.cavity(48, 0.5).instances[0]
    else:
        inst = WL.random_instance(np.random.default_rng(0), 2, (40, 30), 1, (0.02, 1.0))
    for seed in range(4):
        s = gpu_solver([inst], [1.0], [1.0], 64, 64, seed=seed, walk_k=5)
        t = s.autotune(torch.full((inst.ncells,), 0.5, dtype=torch.float64, device="cuda"))
        if kind == "box" or t["refill_lanes"] == 0:
            assert t["walk_k"] == 5
        else:
            assert t["walk_k"] in (5, 8, 16, 32)
