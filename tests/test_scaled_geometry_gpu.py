"""Lengths times a power of two: every FP64 operation of a fixed-step trace scales with them, so positions and times
come out times that power, bit for bit, and directions, weights and step counts as they were."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ck():
    from paper_1209_6038_gb300 import build, cloak
    build.build()
    return cloak


def trace(ck, variant, pol, rays, scale):
    import torch
    c = ck.Cloak(variant, 0.5 * scale, 1.0 * scale, 2.0 * scale).integrator(ck.RK4, 2.0 ** -7 * scale, ck.FP64, 5000)
    r = rays.copy()
    r[:, :3] *= scale
    out = ck.records_to_numpy(c.trace_rays(pol, torch.from_numpy(r))).copy()
    c.close()
    return out


@pytest.mark.parametrize("variant,pol", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("rays", [61, 5003])
@pytest.mark.parametrize("power", [110, 300, -90, -140, -300])
def test_traces_scale_with_the_geometry(ck, variant, pol, rays, power):
    """Eight lanes per ray and one thread per ray; scales on both sides of the integer products' range (2^-127 .. 2^128)
    and of single precision."""
    from paper_1209_6038_gb300 import inputs
    r = inputs.ray_set(rays, 23, "mixed", 1.0, 2.0)
    ref, got = trace(ck, variant, pol, r, 1.0), trace(ck, variant, pol, r, 2.0 ** power)
    for f in ("status", "steps", "mode", "exit_dir", "weight"):
        assert np.array_equal(got[f], ref[f], equal_nan=True), f
    through = np.isin(ref["status"], [1, 2])
    assert through.sum() > rays // 4
    for f in ("exit_pos", "tof"):
        assert np.array_equal(got[f][through], ref[f][through] * 2.0 ** power), f
