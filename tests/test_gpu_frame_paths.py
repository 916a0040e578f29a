"""Frames at the edges of the single-pose kernels' rules (segments side by side
up to eight per block, blur ranges, ray setup in blocks of ten rays): the
batched path, which marches one ray per warp and sets its rays up one per
thread, must give the same bits, and one ray count above each rule the same
values as the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2508_06768_gb300 import inputs as I
from tests.helpers import GRAD_TOL, gpu_grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,bf16,refine", [(0, False, 0), (1, True, 0), (0, True, 1)])
@pytest.mark.parametrize("n_rays,S", [(1, 1), (9, 255), (10, 256), (11, 257), (21, 512), (64, 513), (33, 1025),
                                      (7, 2048), (12, 2049), (5, 4200)])
def test_frame_equals_batch_of_one(n_rays, S, mode, bf16, refine):
    import torch
    from paper_2508_06768_gb300 import binding as B
    from paper_2508_06768_gb300.render import BatchRenderer
    rng = np.random.default_rng(n_rays)
    data = (1.5 + 0.02 * rng.standard_normal((37, 41, 44))).astype(np.float32)
    vol = torch.from_numpy(data).cuda().to(torch.bfloat16 if bf16 else torch.float32)
    fan = I.Fan(n_rays, S, math.radians(64), 0.1 * S ** 0.8, 5.0, 0.5)
    prm = I.Params(seed=11, mode=mode, refine=refine)
    sp, org = (1.0, 0.9, 1.1), (0.25, 0.0, -0.5)
    pose = torch.tensor([21.3, 18.4, 1.2, 0.11, -0.07, 0.4], device="cuda")
    r = BatchRenderer(vol, sp, org, [fan], prm)
    G = torch.from_numpy(rng.standard_normal((n_rays, S)).astype(np.float32)).cuda()
    r.run(pose[None], G.reshape(-1))
    img, valid, status = B.render_fwd(vol, sp, org, pose, fan, prm)
    assert torch.equal(img, r.image(0)) and torch.equal(valid, r.ray_valid)
    assert torch.equal(status, r.status)
    if not refine:      # the refined batch differentiates at the corrected states
        gv, gp, _ = B.render_bwd(vol, sp, org, pose, fan, prm, G)
        assert torch.equal(gv, r.grad_vol) and torch.equal(gp, r.grad_poses[0])
    # the pose-only calls (the march samples dZ/dp) of both paths
    r2 = BatchRenderer(vol, sp, org, [fan], prm)
    B.render_batch(r2.volume, sp, org, pose[None].contiguous(), r2.plan_host, r2.plan_dev, prm, r2.images, r2.workspace,
                   ray_valid=r2.ray_valid, grad_images=G.reshape(-1), grad_poses=r2.grad_poses, status=r2.status)
    if not refine:
        _, gp1, _ = B.render_bwd(vol, sp, org, pose, fan, prm, G, want_vol=False)
        assert torch.equal(gp1, r2.grad_poses[0])


@pytest.mark.parametrize("n_rays", [2432, 2433, 4096, 4097])
def test_ray_counts_around_the_rules(n_rays):
    rng = np.random.default_rng(3)
    vol = I.Volume((1.5 + 0.02 * rng.standard_normal((30, 31, 33))).astype(np.float32))
    fan, prm = I.Fan(n_rays, 300, math.radians(60), 30.0), I.Params(seed=2, mode=1)
    pose = np.array([16.0, 15.0, 0.5, 0.05, 0.1, 0.2], dtype=np.float32)
    G = I.random_weights((n_rays, 300), 8)
    gv, gp = gpu_grad(vol, pose, fan, prm, G)
    rv, rp = oracle.render_grad(vol, pose, fan, prm, G.astype(np.float64))
    assert np.linalg.norm(gv - rv) <= GRAD_TOL * np.linalg.norm(rv)
    assert np.linalg.norm(gp - rp) <= GRAD_TOL * np.linalg.norm(rp)


def test_frame_without_blur_and_with_nonfinite_volume():
    # packed rows of every alignment (no blur), and a volume with NaN, infinite
    # and zero voxels: the same rows are not finite on both paths
    import torch
    from paper_2508_06768_gb300 import binding as B
    from paper_2508_06768_gb300.render import BatchRenderer
    rng = np.random.default_rng(5)
    data = (1.5 + 0.1 * rng.standard_normal((24, 24, 24))).astype(np.float32)
    data[12, 5, 7], data[15, 11, 9], data[9, 12, 12] = np.nan, np.inf, 0.0
    vol = torch.from_numpy(data).cuda()
    for S in (301, 302, 303, 304):
        for atten in (0, 1):
            fan, prm = I.Fan(19, S, math.radians(60), 22.0), I.Params(seed=1, blur=0, atten=atten)
            pose = torch.tensor([11.5, 11.5, 0.5, 0.0, 0.0, 0.3], device="cuda")
            r = BatchRenderer(vol, (1.0,) * 3, (0.0,) * 3, [fan, fan], prm, with_bwd=False)
            r.run(pose[None].repeat(2, 1))
            img, valid, status = B.render_fwd(vol, (1.0,) * 3, (0.0,) * 3, pose, fan, prm)
            a, b = img.cpu().numpy(), r.image(0).cpu().numpy()
            assert np.array_equal(a, b, equal_nan=True)
            assert torch.equal(valid, r.ray_valid[:19])
            n = int(np.count_nonzero(~np.isfinite(a)))
            assert n > 0 and int(status[1]) == n


@pytest.mark.parametrize("mode,bf16,refine", [(0, False, 0), (1, True, 0), (0, False, 1)])
@pytest.mark.parametrize("fans", [[(1, 1), (33, 17)], [(64, 300), (31, 255), (70, 1030)]])
def test_lane_form_forward_alone(fans, mode, bf16, refine):
    # the forward-only kernel of the one-lane-per-ray form keeps nothing, and
    # renders the bits of the call with a backward
    import torch
    from paper_2508_06768_gb300 import binding as B
    from paper_2508_06768_gb300.render import BatchRenderer
    rng = np.random.default_rng(len(fans))
    data = (1.5 + 0.02 * rng.standard_normal((37, 41, 44))).astype(np.float32)
    vol = torch.from_numpy(data).cuda().to(torch.bfloat16 if bf16 else torch.float32)
    fans = [I.Fan(n, s, math.radians(64), 0.1 * s ** 0.8, 5.0, 0.5) for n, s in fans]
    prm = I.Params(seed=11, mode=mode, refine=refine)
    poses = torch.tensor([[21.3, 18.4, 1.2, 0.11, -0.07, 0.4]] * len(fans), device="cuda")
    poses[:, 0] += torch.arange(len(fans), device="cuda")
    a, b = [BatchRenderer(vol, (1.0, 0.9, 1.1), (0.0, 0.0, 0.0), fans, prm, schedule=B.ScheduleDesc(0, 0, 0, 1),
                          with_bwd=w) for w in (False, True)]
    a.run(poses)
    b.run(poses, torch.ones_like(b.images))
    assert torch.equal(a.images, b.images) and torch.equal(a.ray_valid, b.ray_valid)
    assert torch.equal(a.status, b.status)
