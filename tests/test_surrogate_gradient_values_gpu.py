"""The surrogate's batch gradient against values on file (tests/golden/make_surrogate_gradient.py): what a change of the
backward pass may not move, or training from a seed would give another network."""
import os
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")
sys.path.insert(0, GOLDEN)
import make_surrogate_gradient as M  # noqa: E402


def golden(stage, n):
    with open(os.path.join(GOLDEN, "surrogate_gradient.txt")) as f:
        for line in f:
            w = line.split()
            if (int(w[0]), int(w[1])) == (stage, n):
                return np.array([int(v, 16) for v in w[2:]], np.uint32).view(np.float32)
    raise KeyError((stage, n))


@pytest.fixture(scope="module")
def gradient():
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()

    def step(stage, n):
        c = ck.Cloak(ck.RADIAL)
        ck.cloak_surrogate_params(c.h, M.params())
        x, t = M.batch(stage, n)
        g = ck.cloak_surrogate_step(c.h, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), stage=stage, lr=0.0)
        c.close()
        return np.asarray(g, np.float32)[::M.STRIDE]

    return step


@pytest.mark.parametrize("stage,n", M.CASES)
def test_gradient_keeps_its_roundings(gradient, stage, n):
    """Every BF16 activation and dZ rounds as it did: what remains is the order of at most 152 FP32 partial sums, whose
    relative effect is below sqrt(152) 2^-24 = 7.3e-7.  One changed rounding in some hundred thousand dZ is 1e-5."""
    ref = golden(stage, n).astype(np.float64)
    assert np.linalg.norm(gradient(stage, n) - ref) <= 7.3e-7 * np.linalg.norm(ref)


@pytest.mark.parametrize("stage,n", M.CASES)
def test_gradient_sums_in_its_order(gradient, stage, n):
    """Slices are added one after the other and bias columns in their fixed tree: the same bits."""
    assert np.array_equal(gradient(stage, n).view(np.uint32), golden(stage, n).view(np.uint32))
