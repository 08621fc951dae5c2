"""The device forms of the integer double arithmetic (csrc/soft64.cuh: carry chains that the host build does not have)
against the hardware's operations, bit for bit; and the right-hand sides on integer products against the same ones on
hardware products, wherever the range check lets the former stand."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    from paper_1209_6038_gb300 import build
    torch.cuda.init()
    out = str(tmp_path_factory.mktemp("soft64d") / "libs64d.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, "-o", out, os.path.join(HERE, "soft64_device.cu")], check=True)
    return C.CDLL(out)


def doubles(rng, n, lo, hi):
    """Random signs, exponents in [lo, hi]; significands full, short (products tie or are exact), sparse or all ones."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    short = rng.integers(0, 53, n).astype(np.uint64)
    kind = rng.integers(0, 8, n)
    m = np.where(kind < 3, (m >> short) << short, m)
    m = np.where(kind == 3, np.uint64((1 << 52) - 1) << short & np.uint64((1 << 52) - 1), m)
    m = np.where(kind == 4, np.uint64(1) << rng.integers(0, 52, n).astype(np.uint64), m)
    e = rng.integers(lo + 1023, hi + 1024, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


def ptr(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("lo,hi", [(-1, 1), (-127, 127), (-510, 511)])
def test_products(lib, lo, hi):
    import torch
    n = 2_000_003
    rng = np.random.default_rng(hi + 7)
    a, b = (torch.from_numpy(doubles(rng, n, lo, hi)).cuda() for _ in range(2))
    soft, hw = torch.empty_like(a), torch.empty_like(a)
    torch.cuda.synchronize()
    assert lib.s64d_mul(ptr(a), ptr(b), C.c_longlong(n), ptr(soft), ptr(hw)) == 0
    assert torch.equal(soft.view(torch.int64), hw.view(torch.int64))
    assert np.array_equal(hw.cpu().numpy().view(np.uint64), (a * b).cpu().numpy().view(np.uint64))


def test_conversion(lib):
    import torch
    n = 1_000_003
    a = np.abs(doubles(np.random.default_rng(3), n, -140, 140))
    a[:4] = (0.0, np.inf, np.nan, 5e-324)
    x = torch.from_numpy(a).cuda()
    soft, hw = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    ok = torch.empty(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.s64d_float(ptr(x), C.c_longlong(n), ptr(soft), ptr(hw), ptr(ok)) == 0
    inside = torch.from_numpy((a == 0) | ((a >= 2.0 ** -125) & (a < 2.0 ** 127))).cuda()
    assert torch.equal(ok.bool(), inside)
    assert torch.equal(soft[inside].view(torch.int32), hw[inside].view(torch.int32))


@pytest.mark.parametrize("vm", [1, 2, 3])
@pytest.mark.parametrize("power", [0, -40, 40, 100])
def test_right_hand_sides(lib, vm, power):
    """States of the shell and close to r = R1, lengths and velocities times 2^power, with exact zeros among the
    components: where the range check accepts, the accelerations and r^2 are the hardware's (a zero may differ in sign)."""
    import torch
    n = 400_003
    rng = np.random.default_rng(vm)
    r = 0.5 + 0.5 * np.where(rng.uniform(size=n) < 0.5, rng.uniform(0, 1, n), 2.0 ** -rng.uniform(1, 50, n))
    a = rng.uniform(0, 2 * np.pi, n)
    y = np.stack([r * np.cos(a), r * np.sin(a), rng.uniform(-1, 1, n), *(rng.normal(0, 1, (3, n)) * 2.0 ** rng.integers(-20, 3, (3, n)))], 1)
    for k, c in ((3, 5), (5, 1), (7, 3), (11, 4), (13, 0)):
        y[::k, c] = 0.0
    y *= 2.0 ** power
    x = torch.from_numpy(y).cuda()
    soft, hw = (torch.empty((n, 4), dtype=torch.float64, device="cuda") for _ in range(2))
    ok = torch.empty(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.s64d_accel(vm, C.c_double(0.5 * 2.0 ** power), ptr(x), C.c_longlong(n), ptr(soft), ptr(hw), ptr(ok)) == 0
    ok = ok.bool()
    assert power or ok.sum() > n // 3
    assert (soft[ok] == hw[ok]).all()
    nonzero = ok[:, None] & (hw != 0)
    assert torch.equal(soft[nonzero].view(torch.int64), hw[nonzero].view(torch.int64))
