"""The byte offset of a cell in a plane (csrc/plane.cuh, compiled for the host) over the whole range
of lattice sizes that the library accepts: up to 2^31 - 64 cells, where a plane of doubles has
2^34 bytes."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def offset(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plane") / "plane_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC",
                    os.path.join(HERE, "plane_host.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).plane_offset
    f.restype = ctypes.c_ulonglong
    return f


@pytest.mark.parametrize("index", [0, 1, 2**29 - 1, 2**29, 2**29 + 1, 2**30 - 1, 2**30, 2**30 + 7,
                                   2**31 - 65])
@pytest.mark.parametrize("size", [8, 4])
def test_offset_does_not_wrap(offset, index, size):
    assert offset(int(size == 8), index) == index * size
