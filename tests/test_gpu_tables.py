"""Edges of the scan conversion's tiles and image groups, and of the HU map's
lookup table: every form must give the bits of the plain one (one image per
call; the breakpoint search that small volumes take) and match the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2508_06768_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,rays,rows,wh", [(1, 2, 2, (3, 5)), (3, 9, 33, (33, 9)), (9, 8, 32, (32, 8)),
                                                (15, 65, 100, (31, 64)), (16, 17, 257, (100, 33))])
def test_scan_groups_and_tiles(count, rays, rows, wh):
    import torch
    from paper_2508_06768_gb300.render import ScanConverter
    fan = I.Fan(rays, rows, math.radians(75), 40.0)
    conv = ScanConverter(fan, *wh)
    rng = np.random.default_rng(count)
    x = torch.from_numpy(rng.standard_normal((count, rays, rows)).astype(np.float32)).cuda().requires_grad_(True)
    y = conv(x)
    g = torch.from_numpy(rng.standard_normal(tuple(y.shape)).astype(np.float32)).cuda()
    (gx,) = torch.autograd.grad(y, x, g)
    for c in range(count):
        xc = x[c].detach().clone().requires_grad_(True)
        yc = conv(xc)
        assert torch.equal(yc, y[c])
        assert torch.equal(torch.autograd.grad(yc, xc, g[c].clone())[0], gx[c])
    ref = oracle.scan_convert(x[0].detach().cpu().numpy().astype(np.float64), fan, conv.grid)
    refT = oracle.scan_convert_T(g[0].cpu().numpy().astype(np.float64), fan, rays, rows, conv.grid)
    assert np.abs(y[0].detach().cpu().numpy() - ref).max() <= 1e-5
    assert np.linalg.norm(gx[0].cpu().numpy() - refT) <= 1e-5 * max(np.linalg.norm(refT), 1e-30)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("pts", [[0.0], [-3.5, 7.25, 20.0], [-40000.0, -32760.0], [32700.5, 40000.0], [40.0, 41.0]])
def test_hu_table_equals_search(pts, bf16):
    import torch
    from paper_2508_06768_gb300 import binding as B
    rng = np.random.default_rng(len(pts))
    z = np.linspace(1.3, 7.8, len(pts))
    dt = torch.bfloat16 if bf16 else torch.float32
    n = 400003                                  # enough voxels for the table whenever it is small
    mid = int(np.clip(np.mean(pts), -32768, 32767))
    hu = np.clip(rng.integers(mid - 60, mid + 60, n), -32768, 32767)
    hu[:4] = (-32768, 32767, 0, -1)
    h = torch.from_numpy(hu.astype(np.int16)).cuda()
    full = B.hu_to_z(h, pts, z, dtype=dt)
    parts = torch.cat([B.hu_to_z(h[i:i + 800].contiguous(), pts, z, dtype=dt) for i in range(0, n, 80000)])
    whole = torch.cat([full[i:i + 800] for i in range(0, n, 80000)])
    assert torch.equal(parts, whole)
    # an input and an output that 16-byte accesses cannot take
    buf = torch.empty(n + 3, dtype=torch.int16, device="cuda")[3:]
    buf.copy_(h)
    out = torch.empty(n + 1, dtype=dt, device="cuda")[1:]
    assert torch.equal(B.hu_to_z(buf, pts, z, out=out), full)
    ref = np.interp(hu.astype(np.float64), pts, z)
    tol = 2.0 ** -8 if bf16 else 3e-7
    assert np.all(np.abs(full.float().cpu().numpy() - ref) <= np.abs(ref) * tol * 1.01)
