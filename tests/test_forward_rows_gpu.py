"""The surrogate's forward call reads its FP32 rows and writes its outputs in the fused kernel; where the outputs
overlap the inputs the rows go through the padded scratch first.  Both give the same bits, at the edges of a
128-row tile, of a pair of tiles and of a full wave of pairs, and nothing beyond the last row is written."""
import numpy as np
import pytest
import torch

from paper_1209_6038_gb300 import cloak as ck

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 255, 256, 257, 152 * 256 - 1, 152 * 256 + 129])
def test_rows_equal_the_scratch_path(n, fp16):
    c = ck.Cloak(ck.RADIAL)
    rng = np.random.default_rng(n)
    ck.cloak_surrogate_params(c.h, rng.normal(0, 0.1, ck.SUR_NPARAMS).astype(np.float32))
    ck.cloak_surrogate_set_precision(c.h, fp16)
    x = torch.from_numpy(rng.uniform(-1, 1, (n, 7)).astype(np.float32)).cuda()
    y = torch.full((n + 64, 5), 77.0, device="cuda")
    ck.cloak_surrogate_forward(c.h, x, y)
    shared = torch.empty(7 * n, device="cuda")  # outputs over the inputs
    shared.copy_(x.reshape(-1))
    ck.cloak_surrogate_forward(c.h, shared.view(n, 7), shared[:5 * n].view(n, 5))
    torch.cuda.synchronize()
    assert torch.equal(y[:n], shared[:5 * n].view(n, 5))
    assert torch.isfinite(y[:n]).all() and (y[n:] == 77.0).all()
    c.close()
