"""Eight lanes per ray against one thread per ray: the FP64 paths take the same steps whichever way a ray is
integrated -- one thread of a full warp, a group of eight lanes in a call of few rays, a long ray of the queue, or a
ray that its warp finishes in eight lanes after it stepped in one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ck():
    import torch
    from paper_1209_6038_gb300 import build, cloak
    build.build()
    cloak.load()
    torch.cuda.init()
    return cloak


def same(a, b, exact):
    assert np.array_equal(a["status"], b["status"])
    assert np.array_equal(a["steps"], b["steps"])
    assert np.array_equal(a["tile_id"], b["tile_id"])
    # the queue's crossing search rounds its quotients differently (or takes Newton steps): a crossing is found to
    # 1e-13 of a step, a step is shorter than the path, and the path is below 10
    tol = 0.0 if exact else 4e-11
    for f in ("exit_pos", "exit_dir", "tof", "weight"):
        assert np.max(np.abs(a[f] - b[f])) <= tol, f


@pytest.mark.parametrize("variant,pol", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("integ,h", [(0, 2e-3), (1, 1e-9)])
def test_few_rays_step_as_many(ck, variant, pol, integ, h):
    """1, 3, 4, 5 and 61 rays (eight lanes each) against the same rays inside a large call (one thread each)."""
    import torch
    from paper_1209_6038_gb300 import inputs
    rays = torch.from_numpy(inputs.ray_set(20000, 11, "mixed"))
    c = ck.Cloak(variant).integrator(integ, h)
    many = ck.records_to_numpy(c.trace_rays(pol, rays))
    for n in (1, 3, 4, 5, 61):
        first = 17 * n
        same(ck.records_to_numpy(c.trace_rays(pol, rays[first:first + n])), many[first:first + n], True)
    c.close()


@pytest.mark.parametrize("variant,pol", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("integ,h", [(0, 2e-3), (1, 1e-9)])
@pytest.mark.parametrize("blocks", [0, 4])
def test_queued_rays_step_as_plain_ones(ck, variant, pol, integ, h, blocks):
    """The queue with and without long-ray blocks: rays start in eight lanes, or change to them when four or fewer
    are left in a warp; the plain path of this size keeps one thread per ray."""
    from paper_1209_6038_gb300 import inputs
    eye, target, up = inputs.camera_pose(20.0, 33.0)
    c = ck.Cloak(variant).integrator(integ, h).camera(eye, target, up, 60.0, 321, 181)
    plain = ck.records_to_numpy(c.render_records(pol, 1, 5))
    c.schedule(ck.SCHED_WAVEFRONT)
    ck.cloak_set_schedule_tuning(c.h, blocks, 1, 4.0)
    same(ck.records_to_numpy(c.render_records(pol, 1, 5)), plain, False)
    c.close()
