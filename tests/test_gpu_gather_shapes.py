"""Volume gradient at the edges of the gather's tiling: volumes whose last
brick holds one voxel, a few or all eight, an output the vector stores cannot
take, and ray counts on both sides of every unit size."""
import math

import numpy as np
import pytest

import oracle
from paper_2508_06768_gb300 import inputs as I
from tests.helpers import GRAD_TOL, gpu_grad

pytestmark = pytest.mark.gpu


def _volume(shape_xyz, seed):
    nx, ny, nz = shape_xyz
    rng = np.random.default_rng(seed)
    return I.Volume((1.5 + 0.1 * rng.standard_normal((nz, ny, nx))).astype(np.float32))


def _pose(shape_xyz):
    return np.array([0.5 * (shape_xyz[0] - 1) + 0.13, 0.5 * (shape_xyz[1] - 1) - 0.21, 0.4, 0.21, -0.17, 0.3],
                    dtype=np.float32)


@pytest.mark.parametrize("shape", [(2, 2, 2), (5, 9, 10), (61, 12, 17), (64, 9, 8), (65, 8, 33), (66, 17, 16)])
def test_volume_gradient_at_brick_edges(shape):
    import torch
    from paper_2508_06768_gb300 import binding as B
    vol, pose, prm = _volume(shape, 5), _pose(shape), I.Params(seed=2, mode=1)
    fan = I.Fan(37, 203, math.radians(70), 31.0)
    G = I.random_weights((fan.n_rays, fan.n_samples), 3)
    gv, gp = gpu_grad(vol, pose, fan, prm, G)
    rv, rp = oracle.render_grad(vol, pose, fan, prm, G.astype(np.float64))
    assert np.linalg.norm(gv - rv) <= GRAD_TOL * np.linalg.norm(rv)
    assert np.linalg.norm(gp - rp) <= GRAD_TOL * np.linalg.norm(rp)
    # an output that is not 16-byte aligned gets the same bits
    n = int(np.prod(shape))
    out = torch.full((n + 1,), float("nan"), device="cuda")[1:].view(*vol.data.shape)
    B.render_bwd(torch.from_numpy(vol.data).cuda(), vol.spacing, vol.origin, torch.from_numpy(pose).cuda(), fan, prm,
                 torch.from_numpy(G).cuda(), grad_vol=out)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), gv)


@pytest.mark.parametrize("n_rays", [1, 31, 33, 4001, 20001, 160001, 330001, 640001])
def test_volume_gradient_for_every_unit_size(n_rays):
    shape = (40, 40, 40)
    vol, pose, prm = _volume(shape, 6), _pose(shape), I.Params(seed=3, mode=1)
    fan = I.Fan(n_rays, 3, math.radians(60), 20.0)
    G = I.random_weights((n_rays, 3), 4)
    gv, gp = gpu_grad(vol, pose, fan, prm, G)
    rv, rp = oracle.render_grad(vol, pose, fan, prm, G.astype(np.float64))
    assert np.linalg.norm(gv - rv) <= GRAD_TOL * np.linalg.norm(rv)
    assert np.linalg.norm(gp - rp) <= GRAD_TOL * np.linalg.norm(rp)


@pytest.mark.parametrize("n_rays", [5, 700])
def test_volume_gradient_of_rays_through_many_bricks(n_rays):
    # 275 bricks along x: more changes per ray than the warp-per-ray run pass takes
    shape = (2200, 3, 3)
    vol, prm = _volume(shape, 7), I.Params(seed=4, mode=1)
    pose = np.array([3.3, 1.1, 0.9, 0.0, math.pi / 2, 0.0], dtype=np.float32)   # beam along +x
    fan = I.Fan(n_rays, 400, 1e-3, 2190.0, 0.0, 0.0)
    G = I.random_weights((n_rays, 400), 5)
    gv, gp = gpu_grad(vol, pose, fan, prm, G)
    rv, rp = oracle.render_grad(vol, pose, fan, prm, G.astype(np.float64))
    assert np.linalg.norm(gv - rv) <= GRAD_TOL * np.linalg.norm(rv)


def test_volume_gradient_of_a_volume_of_many_bricks():
    # 640 x 360 x 360 voxels: over 65536 bricks, whose counts are summed in two steps
    shape = (640, 360, 360)
    rng = np.random.default_rng(8)
    vol = I.Volume((1.5 + 0.1 * rng.standard_normal((360, 360, 640), dtype=np.float32)))
    prm, fan = I.Params(seed=5, mode=1), I.Fan(40, 500, math.radians(60), 250.0)
    pose = np.array([560.0, 310.0, 300.0, 0.4, 3.3, 0.2], dtype=np.float32)
    G = I.random_weights((fan.n_rays, fan.n_samples), 6)
    gv, gp = gpu_grad(vol, pose, fan, prm, G)
    rv, rp = oracle.render_grad(vol, pose, fan, prm, G.astype(np.float64))
    assert np.linalg.norm(gv - rv) <= GRAD_TOL * np.linalg.norm(rv)
    assert np.linalg.norm(gp - rp) <= GRAD_TOL * np.linalg.norm(rp)
