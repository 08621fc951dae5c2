"""Camera rays close to the cylinder's outline, where FP32 has to leave the decision to FP64: whole images of the queued and
batched renders, hitting pixels included, against the plain schedule, whose entry search is FP64 throughout."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def outline(R2, H, distance, elevation, where, fov):
    """Eye at the given distance, looking at a point of the outline: the side at mid-height, the rim of the top face on
    the near or far side, the corner where the side meets the rim, or the cylinder's middle."""
    e = math.radians(elevation)
    eye = np.array([distance * math.cos(e), 0.1 * R2, distance * math.sin(e)])
    az = math.atan2(eye[1], eye[0])
    d = math.hypot(eye[0], eye[1])
    t = az + math.acos(min(1.0, R2 / d)) if d > R2 else az  # the tangent point seen from the eye
    target = {"side": (R2 * math.cos(t), R2 * math.sin(t), 0.1 * H),
              "near": (R2 * math.cos(az), R2 * math.sin(az), 0.5 * H),
              "far": (-R2 * math.cos(az), -R2 * math.sin(az), 0.5 * H),
              "corner": (R2 * math.cos(t), R2 * math.sin(t), 0.5 * H),
              "middle": (0.0, 0.0, 0.0)}[where]
    return tuple(eye), tuple(float(v) for v in target), fov


CASES = [(1.0, 2.0, 5.0, 0.0, "side", 60.0), (1.0, 2.0, 5.0, 0.0, "side", 0.01), (1.0, 2.0, 5.0, 20.0, "side", 1e-4),
         (1.0, 2.0, 5.0, 20.0, "corner", 0.1), (1.0, 2.0, 5.0, 45.0, "far", 1.0), (1.0, 2.0, 5.0, 10.0, "near", 0.05),
         (1.0, 2.0, 60.0, 5.0, "side", 0.5), (1.0, 2.0, 300.0, 30.0, "middle", 1.0), (1.0, 2.0, 1.02, 0.0, "side", 30.0),
         (0.03, 2.0, 5.0, 20.0, "middle", 2.0), (3.0, 0.05, 5.0, 3.0, "near", 5.0), (0.7, 9.0, 4.0, 60.0, "corner", 3.0),
         (1.0, 2.0, 5.0, 89.9, "far", 20.0)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("width,height,spp", [(96, 71, 1), (41, 33, 5)])
def test_images_at_the_outline(case, width, height, spp):
    """The same rays take the same steps on both schedules; crossings agree to 1e-13 of a step, so colours and weights to
    single precision."""
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    R2, H, distance, elevation, where, fov = case
    eye, target, fov = outline(R2, H, distance, elevation, where, fov)
    c = ck.Cloak(ck.AZIMUTHAL, 0.5 * R2, R2, H).integrator(ck.DP45, 1e-6, ck.FP64, 2000)
    c.camera(eye, target, (0, 0, 1), fov, width, height)
    plain = c.render(1, spp, 3).cpu().numpy()
    status = ck.records_to_numpy(c.render_records(1, spp, 3))["status"]
    assert (status == 0).any() and (status != 0).any()  # the outline is in the picture
    c.schedule(ck.SCHED_WAVEFRONT)
    queued = c.render(1, spp, 3).cpu().numpy()
    batch = torch.empty((height, width, 4), device="cuda")
    ck.cloak_render_batch(c.h, [(1, 1, eye, target, (0, 0, 1), fov, batch)], spp, 3)
    c.close()
    assert np.abs(queued - plain).max() <= 1e-6
    assert np.abs(batch.cpu().numpy() - plain).max() <= 1e-6
