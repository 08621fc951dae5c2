"""The correctly rounded double products of the FP64 integrator (csrc/soft64.cuh): the host build against IEEE
arithmetic bit for bit, and on the GPU the right-hand sides that use them, inside and outside their range,
against extended precision."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1209_6038_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("soft64") / "libs64h.so")
    subprocess.run(["g++", "-O2", "-fPIC", "-shared", "-I", CSRC, "-x", "c++", "-o", out,
                    os.path.join(HERE, "soft64_host.cpp")], check=True)
    L = C.CDLL(out)
    L.s64h_mul.argtypes, L.s64h_mul.restype = [C.c_double] * 2, C.c_double
    L.s64h_in_range.argtypes, L.s64h_in_range.restype = [C.c_double], C.c_int
    L.s64h_to_float.argtypes, L.s64h_to_float.restype = [C.c_double, C.POINTER(C.c_int)], C.c_float
    L.s64h_from_float.argtypes, L.s64h_from_float.restype = [C.c_float], C.c_double
    return L


def samples(rng, n, lo, hi):
    """Doubles of random sign, exponents in [lo, hi], significands full, short (products tie), or all ones."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    short = rng.integers(0, 53, n).astype(np.uint64)
    m = np.where(rng.uniform(size=n) < 0.5, m, (m >> short) << short)
    m = np.where(rng.uniform(size=n) < 0.02, np.uint64((1 << 52) - 1), m)
    e = rng.integers(lo + 1023, hi + 1024, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


@pytest.mark.parametrize("lo,hi", [(-1, 1), (-127, 127), (-500, 500)])
def test_products_round_as_ieee(lib, lo, hi):
    rng = np.random.default_rng(hi)
    a, b = samples(rng, 40000, lo, hi), samples(rng, 40000, lo, hi)
    got = np.array([lib.s64h_mul(x, y) for x, y in zip(a.tolist(), b.tolist())])
    assert np.array_equal(got.view(np.uint64), (a * b).view(np.uint64))


@pytest.mark.parametrize("value,inside", [(2.0 ** -127, 1), (-1.0, 1), (np.nextafter(2.0 ** 128, 0), 1), (0.0, 0),
                                          (-0.0, 0), (np.nextafter(2.0 ** -127, 0), 0), (2.0 ** 128, 0), (5e-324, 0),
                                          (np.inf, 0), (-np.inf, 0), (np.nan, 0)])
def test_range(lib, value, inside):
    assert lib.s64h_in_range(float(value)) == inside


def test_conversions(lib):
    rng = np.random.default_rng(3)
    ok = C.c_int()
    for v in np.concatenate([np.abs(samples(rng, 20000, -124, 125)), [0.0]]).tolist():
        f = lib.s64h_to_float(v, C.byref(ok))
        assert ok.value == 1 and f == float(np.float32(v))
        if f > 0:
            assert lib.s64h_from_float(f) == f
    for v in (2.0 ** -126, 2.0 ** 127, 5e-324, np.inf, np.nan):
        lib.s64h_to_float(float(v), C.byref(ok))
        assert ok.value == 0


def reference(variant, pol, R1, y):
    """dv/dt in extended precision: the closed cylindrical form, M = diag(K, f, f) or diag(K, f, K)."""
    y = y.astype(np.longdouble)
    x, v = y[:, :3], y[:, 3:]
    r = np.hypot(x[:, 0], x[:, 1])
    c, s = x[:, 0] / r, x[:, 1] / r
    vr, vt, vz = v[:, 0] * c + v[:, 1] * s, v[:, 1] * c - v[:, 0] * s, v[:, 2]
    u = r - np.longdouble(R1)
    g = 2 * np.longdouble(R1) / (r * u)
    if pol == 0:
        ar, at, az = g / 2 * (vt * vt + vz * vz - vr * vr), -g * vr * vt, -g * vr * vz
    elif variant == 0:
        ar, at, az = R1 * (u * vz * vz - r * vt * vt) / r ** 3, -g * vr * vt, -g * vr * vz
    else:
        ar, at, az = -R1 * vt * vt / r ** 2, -g * vr * vt, 0 * vz
    return np.stack([ar * c - at * s, ar * s + at * c, az], 1), np.abs(g) * (v ** 2).sum(1) + np.abs(ar)


@pytest.mark.gpu
@pytest.mark.parametrize("variant,pol", [(0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -120, 2.0 ** -140, 2.0 ** 140])
def test_right_hand_sides_in_and_out_of_range(variant, pol, scale):
    """Lengths and velocities times scale: 2^-140 and 2^140 lie outside the integer products' range and take the
    hardware's; exact zeros (in-plane velocities, points on an axis) do so at every scale.  Tolerance: some forty
    roundings of 2^-53 relative to the largest term, and the cancellation of u = r - R1 <= r, u >= 0.02 r here."""
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    rng = np.random.default_rng(7)
    n = 1003
    R1, R2 = 0.5 * scale, 1.0 * scale
    r, a = rng.uniform(0.52, 1.0, n), rng.uniform(0, 2 * np.pi, n)
    y = np.concatenate([np.stack([r * np.cos(a), r * np.sin(a), rng.uniform(-1, 1, n)], 1), rng.normal(0, 1, (n, 3))],
                       1) * scale
    y[::3, 5] = 0.0
    y[::5, 1] = 0.0
    y[1::7, 3] = 0.0
    y[2::9, 4] = 0.0
    c = ck.Cloak(variant, R1, R2, 2.0 * scale)
    d = c.eval_rhs(pol, torch.from_numpy(y)).cpu().numpy()
    c.close()
    ref, size = reference(variant, pol, R1, y)
    assert np.array_equal(d[:, :3], y[:, 3:])
    err = np.abs(d[:, 3:] - ref).max(1)
    assert (err <= 60 * 50 * 2.0 ** -53 * size).all(), (err / size).max()
