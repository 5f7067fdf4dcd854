"""The status reported for the device error word, compiled from its header with the host compiler: a
barrier of the correction solve that gave up is a device failure, not a solve that reached its
iteration cap (whose bit and counts it sets as well), and it is reported once."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_09465_gb300", "csrc")
SHIM = """#include "%s/error_word.h"
extern "C" int status(int e, const char** t) { return iugkp::error_word_status(e, t); }
extern "C" int after(int e) { return iugkp::error_word_after_correction(e); }
"""
BUDGET, RANGE, PCG, WAIT, DEFER = 1, 2, 4, 8, 16
OK, ENOCONV, EBUDGET, EDEVICE = 0, 4, 5, 6


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("word")
    (d / "shim.cpp").write_text(SHIM % CSRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("word,want,part", [(0, OK, ""), (WAIT, EDEVICE, "waited"), (WAIT | PCG, EDEVICE, "waited"),
                                            (WAIT | PCG | BUDGET, EDEVICE, "waited"), (PCG, ENOCONV, "cg_maxit"),
                                            (BUDGET | PCG, EBUDGET, "budget"), (DEFER, EDEVICE, "queue"),
                                            (RANGE, EDEVICE, "check failed")])
def test_status(lib, word, want, part):
    text = ctypes.c_char_p()
    assert lib.status(word, ctypes.byref(text)) == want
    assert part in text.value.decode()


@pytest.mark.parametrize("word", range(32))
def test_a_reported_correction_leaves_only_the_sweeps_bits(lib, word):
    assert lib.after(word) == word & (BUDGET | RANGE | DEFER)
