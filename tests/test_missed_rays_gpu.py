"""Camera rays that miss, decided in FP32: the image's samples against the records of the same rays, whose FP64
entry search and room lookup decide for themselves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# eye, target, field of view: the usual pose; above and beside the cylinder; close to it, inside the shell, on its
# axis; outside the room; along a wall
CAMERAS = [((4.7, 1.7, 0.3), (0, 0, 0), 60.0), ((0.3, 0.2, 6.0), (0, 0, 0), 40.0), ((1.5, 0.1, 0.9), (0, 0, 0), 170.0),
           ((1.0001, 0.0, 0.0), (5, 1, 0.2), 120.0), ((0.7, 0.1, 0.2), (3, 1, 0), 90.0), ((0.0, 0.0, 3.0), (0.1, 0, 0), 60.0),
           ((30.0, 20.0, 5.0), (0, 0, 2), 30.0), ((9.9999, -9.0, 1.0), (9.9999, 9.0, 1.1), 60.0)]


@pytest.mark.parametrize("eye,target,fov", CAMERAS)
@pytest.mark.parametrize("width,height,spp", [(67, 45, 3), (1, 1, 1), (130, 9, 1)])
def test_missed_samples_have_their_rays_colour(eye, target, fov, width, height, spp):
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    c = ck.Cloak(ck.AZIMUTHAL).integrator(ck.DP45, 1e-6, ck.FP64, 2000).schedule(ck.SCHED_WAVEFRONT)
    c.camera(eye, target, (0, 0, 1), fov, width, height)
    img = c.render(1, spp, 3).cpu().numpy().reshape(-1, 4)
    recs = ck.records_to_numpy(c.render_records(1, spp, 3)).reshape(-1, spp)
    # the room's colour of every missed ray, from the panel without the cylinder
    room = c.panel(ck.PANEL_ROOM, spp, 3).cpu().numpy().reshape(-1, 4)
    missed = (recs["status"] == 0).all(1)
    assert np.array_equal(img[missed], room[missed])
    batch = torch.empty((height, width, 4), device="cuda")
    ck.cloak_render_batch(c.h, [(1, 1, eye, target, (0, 0, 1), fov, batch)], spp, 3)
    assert np.array_equal(batch.cpu().numpy().reshape(-1, 4)[missed], room[missed])
    c.close()
