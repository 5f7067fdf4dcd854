"""The step budget with FP64 tracking: a particle of more null candidates than it allows is dropped
and the call fails with EBUDGET, in the landing sweep of the steady loop as in the full sweep. Cell 1
accepts one candidate in 10^17 and a flight through it has 10^14: without the limit its particles
would be followed for hours. (The budget's 2^24 candidates one after the other in FP64: 25 s.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_09465_gb300 import workloads as WL  # noqa: E402
from paper_2506_09465_gb300._lib import IugkpError  # noqa: E402
from gpu_helpers import gpu_solver  # noqa: E402


def test_endless_chains_are_dropped():
    inst = WL.Instance(1, (2, 1, 1), (1.0, 1.0, 1.0), np.array([[1e-14, 1e3]]), np.array([1.0, 0.0]))
    one = np.array([1.0])
    s = gpu_solver([inst], one, one, 4, 4, seed=1, precision=0, tally=0, newton=0, use_graphs=0)
    x = torch.ones(2, dtype=torch.float64, device="cuda")
    with pytest.raises(IugkpError, match="EBUDGET"):
        s.solve_steady(x, 0.0, 1, raise_on_noconv=False)
