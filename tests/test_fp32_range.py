"""The rules that keep FP32 positions out of the sweeps where they do not hold, compiled from their
own header with the host compiler: a candidate whose position or bound has left FP32 counts as near
a face (its cell is not used), and only lengths well inside FP32 are taken for the filtered FP64
sweep."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_09465_gb300", "csrc", "fp32_range.h")
SHIM = """#include "%s"
extern "C" int near_face(float fr, float om, float tol) { return iugkp::face_near(fr, om, tol); }
extern "C" int length_ok(double x) { return iugkp::fp32_length(x); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("range")
    (d / "shim.cpp").write_text(SHIM % HEADER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    so = ctypes.CDLL(str(d / "shim.so"))
    so.near_face.argtypes = [ctypes.c_float] * 3
    so.length_ok.argtypes = [ctypes.c_double]
    return so


def position(g, D, eD, xi):
    """Position, bound, fraction and its complement as the landing sweeps form them, in FP32."""
    f = np.float32
    with np.errstate(all="ignore"):
        X = f(f(g) * f(D) + f(xi))
        tol = f(abs(f(g)) * f(f(D) * f(2.0 ** -20) + f(eD)) + f(2.0 ** -22))
        fr = f(X - np.floor(X))
        return X, tol, fr, f(f(1.0) - fr)


@pytest.mark.parametrize("vtm", [1e39, 1e300, np.inf])
@pytest.mark.parametrize("g", [3.0, -50.0, 0.0])
def test_positions_beyond_fp32_are_near(lib, vtm, g):
    with np.errstate(over="ignore"):
        D = np.float32(vtm)
    X, tol, fr, om = position(g, D, D * np.float32(2.0 ** -20), 0.25)
    assert not np.isfinite(D)
    assert not (X - 50.0 > tol) and not (0.0 - X > tol)  # no wall test tells them
    assert lib.near_face(fr, om, tol) == 1


@pytest.mark.parametrize("fr,tol,near", [(0.5, 0.1, 0), (0.05, 0.1, 1), (0.95, 0.1, 1), (0.1, 0.1, 1), (0.5, 0.5, 1),
                                         (0.0, 0.0, 1), (float("nan"), 0.1, 1), (0.5, float("nan"), 1), (0.5, float("inf"), 1)])
def test_near_inside_fp32(lib, fr, tol, near):
    fr = np.float32(fr)
    assert lib.near_face(fr, np.float32(1.0) - fr, np.float32(tol)) == near


@pytest.mark.parametrize("x,ok", [(1.0, 1), (1e-12, 1), (5e3, 1), (2.0 ** 60, 1), (2.0 ** -60, 1), (2.0 ** 61, 0), (2.0 ** -61, 0),
                                  (1e39, 0), (1e300, 0), (1e-40, 0), (0.0, 0), (float("inf"), 0), (float("nan"), 0)])
def test_lengths_taken(lib, x, ok):
    assert lib.length_ok(x) == ok
