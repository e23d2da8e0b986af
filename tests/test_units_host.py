"""Populations of either sign in integer units (csrc/fixed.cuh, floor58), compiled for the host,
against exact integers: rounded down at every scale, and equal to unit58 for positive values."""
import ctypes
import os
import subprocess
from fractions import Fraction
from math import floor

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("units") / "units_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC",
                    os.path.join(HERE, "units_host.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("top", [1023, 1019, 1060, 300, 1900])
def test_floor58(lib, top):
    rng = np.random.default_rng(top)
    scale = 2.0 ** (top - 1023)                       # value 2^(1023 - top) is below 2
    v = rng.uniform(-2, 2, 3000) * np.exp2(-rng.uniform(0, 62, 3000))
    v[:6] = 1.0, -1.0, -0.5, 2.0 - 2.0**-52, -(2.0 - 2.0**-52), -(2.0**-58)
    v = v * scale
    out = np.empty(len(v), np.int64)
    lib.fx_floor58(v.ctypes.data_as(ctypes.c_void_p), top, out.ctypes.data_as(ctypes.c_void_p),
                   ctypes.c_longlong(len(v)))
    f = Fraction(2) ** (1023 - top + 58)
    exact = [floor(Fraction(float(x)) * f) for x in v]
    assert [int(x) for x in out] == exact
