"""A crossing search that ends at the start of its step: a ray whose step starts behind the metal surface, as rounding can
put it (the mixed queue keeps 48 bits of a position), has no trial point before the surface and ends where it started."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    from paper_1209_6038_gb300 import build
    torch.cuda.init()
    out = str(tmp_path_factory.mktemp("lane") / "liblane.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, "-o", out, os.path.join(HERE, "lane_device.cu")], check=True)
    L = C.CDLL(out)
    L.lane_trace.argtypes = [C.c_int, C.c_int] + [C.c_double] * 4 + [C.c_int, C.POINTER(C.c_double), C.POINTER(C.c_double)]
    return L


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("newton", [0, 1])
@pytest.mark.parametrize("vm", [1, 3])
@pytest.mark.parametrize("depth", [2.0 ** -20, 2.0 ** -30, 2.0 ** -44])
def test_search_that_ends_at_its_start(lib, kind, newton, vm, depth):
    """Extraordinary rays straight towards the axis (no acceleration on that line), from inside R1: SINGULAR there."""
    start = [0.5 * (1 - depth), 0.0, 0.25, -0.5, 0.0, 0.0]
    y = (C.c_double * 6)(*start)
    t = C.c_double(-1.0)
    assert lib.lane_trace(kind, vm, 0.5, 1.0, 2.0, 1e-9, newton, y, C.byref(t)) == 6
    assert np.array_equal(np.array(y[:]), start)
    assert t.value == 0.0
