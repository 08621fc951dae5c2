"""Comparisons of doubles by their bits (csrc/soft64.cuh) against IEEE comparisons, NaNs of both signs, zeros,
infinities and subnormals among them; and a ray whose state becomes NaN."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1209_6038_gb300", "csrc")
NANS = [0x7FF8000000000000, 0x7FFFFFFFFFFFFFFF, 0x7FF0000000000001, 0xFFF8000000000000, 0xFFFFFFFFFFFFFFFF,
        0xFFF0000000000001]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("soft64c") / "libs64c.so")
    subprocess.run(["g++", "-O2", "-fPIC", "-shared", "-I", CSRC, "-x", "c++", "-o", out,
                    os.path.join(HERE, "soft64_compare_host.cpp")], check=True)
    L = C.CDLL(out)
    for f in ("le_pos", "gt_pos"):
        getattr(L, "s64c_" + f).argtypes = [C.c_double] * 2
    for f in ("positive", "not_positive", "not_negative", "isnan", "is_zero", "truncate"):
        getattr(L, "s64c_" + f).argtypes = [C.c_double]
    L.s64c_truncate.restype = C.c_float
    return L


def values():
    pos = [5e-324, 2.2250738585072014e-308, np.nextafter(2.2250738585072014e-308, 0), 1e-300, 0.25, np.nextafter(0.25, 1),
           1.0, 4e-16, 1e300, np.finfo(float).max, np.inf]
    nans = np.array(NANS, np.uint64).view(np.float64)
    return np.array([0.0] + pos), nans


def test_ordering_of_sizes(lib):
    """a <= b and a > b for sizes and NaNs in either place."""
    pos, nans = values()
    for a in np.concatenate([pos, nans]).tolist():
        for b in np.concatenate([pos, nans]).tolist():
            assert bool(lib.s64c_le_pos(a, b)) == (a <= b), (a, b)
            assert bool(lib.s64c_gt_pos(a, b)) == (a > b), (a, b)


def test_signs(lib):
    pos, nans = values()
    for a in np.concatenate([pos, -pos, nans]).tolist():
        assert bool(lib.s64c_positive(a)) == (a > 0), a
        assert bool(lib.s64c_not_positive(a)) == (a <= 0), a
        assert bool(lib.s64c_not_negative(a)) == (a >= 0), a
        assert bool(lib.s64c_isnan(a)) == (a != a), a
        assert bool(lib.s64c_is_zero(a)) == (a == 0), a


def test_truncation(lib):
    """Towards zero, below one unit of the 24 bits, for 2^-125 <= |a| < 2^127; 0 or huge outside."""
    rng = np.random.default_rng(5)
    a = rng.uniform(1, 2, 20000) * 2.0 ** rng.integers(-125, 127, 20000) * rng.choice([-1.0, 1.0], 20000)
    a = np.concatenate([a, [2.0 ** -125, np.nextafter(2.0 ** 127, 0), np.nextafter(1.0, 0), -np.nextafter(2.0, 0)]])
    for v in a.tolist():
        t = lib.s64c_truncate(v)
        assert abs(t) <= abs(v) and abs(v - t) < 2.0 ** -23 * abs(v) and (t > 0) == (v > 0)
    for v in (0.0, 5e-324, np.nextafter(2.0 ** -125, 0)):
        assert lib.s64c_truncate(float(v)) == 0.0 and lib.s64c_truncate(-float(v)) == 0.0
    for v in (2.0 ** 127, 1e300, np.inf):
        assert lib.s64c_truncate(float(v)) >= 2.0 ** 126 and lib.s64c_truncate(-float(v)) <= -(2.0 ** 126)


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("rays", [1, 5000])
def test_a_state_of_nans_crosses_nothing(variant, rays):
    """An extraordinary ray aimed at the axis reaches r = R1 in a whole number of RK4 steps of 1/64: its state is NaN from
    then on, and it ends at the step limit -- alone (eight lanes), among many (one thread), and in the queue."""
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    c = ck.Cloak(variant).integrator(ck.RK4, 1.0 / 64, ck.FP64, 300)
    r = torch.tensor([2.0, 0, 0, -1, 0, 0], dtype=torch.float64).repeat(rays, 1)
    recs = ck.records_to_numpy(c.trace_rays(1, r))
    assert (recs["status"] == 5).all() and (recs["steps"] == 300).all()
    c.camera((5, 0, 0), (0, 0, 0), (0, 0, 1), 60.0, 1, 1).schedule(ck.SCHED_WAVEFRONT)
    queued = ck.records_to_numpy(c.render_records(1, 1, 0))
    assert queued["status"][0] == 5 and queued["steps"][0] == 300
    c.close()
