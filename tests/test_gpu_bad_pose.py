"""Poses that are not finite (device data that nothing refuses, such as a
diverged optimiser's): the probe lies outside the volume and sees no interface,
its pose gradient is NaN, and no other pose of the batch changes."""
import math

import numpy as np
import pytest

from paper_2508_06768_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SP, ORG = (1.0, 0.9, 1.1), (0.25, 0.0, -0.5)


def _setup(n_rays, S):
    import torch
    rng = np.random.default_rng(7)
    data = (1.5 + 0.02 * rng.standard_normal((37, 41, 44))).astype(np.float32)
    fan = I.Fan(n_rays, S, math.radians(64), 40.0, 5.0, 0.5)
    pose = torch.tensor([21.3, 18.4, 1.2, 0.11, -0.07, 0.4], device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    G = torch.randn((n_rays, S), device="cuda", generator=g)
    return torch.from_numpy(data).cuda(), fan, pose, G


# the run pass by rank, by radix with a warp per ray, and with a thread per ray
@pytest.mark.parametrize("n_rays", [5, 2100, 50001])
@pytest.mark.parametrize("angle", [math.nan, math.inf])
def test_frame_of_a_pose_that_is_not_finite(n_rays, angle):
    import torch
    from paper_2508_06768_gb300 import binding as B
    vol, fan, pose, G = _setup(n_rays, 1031)
    prm = I.Params(seed=3, mode=1)
    pose[4] = angle
    img, valid, status = B.render_fwd(vol, SP, ORG, pose, fan, prm)
    gv, gp, st = B.render_bwd(vol, SP, ORG, pose, fan, prm, G)
    assert torch.all(img == 0) and torch.all(valid == fan.n_samples) and not status.any() and not st.any()
    assert torch.isnan(gp[3:]).all() and torch.isfinite(gv).all()
    _, gp, _ = B.render_bwd(vol, SP, ORG, pose, fan, prm, G, want_vol=False)
    assert torch.isnan(gp[3:]).all()


@pytest.mark.parametrize("bad", [{4: math.nan}, {3: math.inf}, {0: math.nan}, {1: -math.inf}, {2: 3e38, 5: math.nan}])
@pytest.mark.parametrize("form", [0, 1])
def test_batch_with_a_pose_that_is_not_finite(bad, form):
    import torch
    from paper_2508_06768_gb300 import binding as B
    from paper_2508_06768_gb300.render import BatchRenderer
    vol, fan, pose, G = _setup(9, 1100)
    prm, sched = I.Params(seed=3, mode=1), B.ScheduleDesc(0, 0, 0, form)
    r = BatchRenderer(vol, SP, ORG, [fan] * 3, prm, schedule=sched)
    poses = torch.stack([pose, pose + 0.01, pose - 0.01])
    r.run(poses, G.repeat(3, 1).reshape(-1))
    ref = [r.image(p).clone() for p in (0, 2)], r.grad_poses.clone()
    for a, x in bad.items():
        poses[1, a] = x
    r.run(poses, G.repeat(3, 1).reshape(-1))
    for p, im in zip((0, 2), ref[0]):
        assert torch.equal(r.image(p), im) and torch.equal(r.grad_poses[p], ref[1][p])
    assert torch.isfinite(r.grad_vol).all() and torch.isfinite(r.images).all()
    if form == 0:
        img, _, _ = B.render_fwd(vol, SP, ORG, poses[1].contiguous(), fan, prm, pose_ctr=1)
        assert torch.equal(img, r.image(1))
