"""Values of the surrogate's batch gradients for test_surrogate_gradient_values_gpu.py (one GB300):

    python tests/golden/make_surrogate_gradient.py > tests/golden/surrogate_gradient.txt

The file in the tree comes from the backward pass with tanhf in the GELU's derivative and weight-gradient slices
added one after the other.  A line: stage, rows, the bits of every 997th component of the gradient (flat FP32 layout of
cloak_surrogate_params)."""
import math
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__)))))
DIMS = (7, 256, 256, 256, 256, 5)
STRIDE = 997
# one chunk of rows per slice; slices of several chunks; the training batch; a row count whose slices are few and long
CASES = ((1, 256), (2, 256), (1, 2560), (1, 19456), (1, 128 * 211), (2, 4864))


def params():
    """Parameters at unit gain: per layer W (out x in), then b."""
    rng = np.random.default_rng(41)
    ps = []
    for a, b in zip(DIMS[:-1], DIMS[1:]):
        ps += [rng.normal(0, 1.0 / math.sqrt(a), (b, a)).ravel(), rng.normal(0, 0.05, b)]
    return np.concatenate(ps).astype(np.float32)


def batch(stage, n):
    """Inputs and targets (t0..t3, confidence target, mask, two spare)."""
    rng = np.random.default_rng([stage, n])
    x = rng.uniform(-1, 1, (n, 7)).astype(np.float32)
    t = np.zeros((n, 8), np.float32)
    t[:, :5] = rng.normal(0, 1, (n, 5))
    t[:, 5] = rng.uniform(0, 1, n) < 0.8
    return x, t


def main():
    import torch

    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    for stage, n in CASES:
        c = ck.Cloak(ck.RADIAL)
        ck.cloak_surrogate_params(c.h, params())
        x, t = batch(stage, n)
        g = ck.cloak_surrogate_step(c.h, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), stage=stage, lr=0.0)
        c.close()
        print(stage, n, *(f"{v:08x}" for v in np.asarray(g, np.float32)[::STRIDE].view(np.uint32)))


if __name__ == "__main__":
    main()
