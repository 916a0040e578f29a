"""Every size of image group in the scan conversion, on displays of few and of
many tiles, narrow and wide: each image of a call gets the bits of a call of its
own, and the values of the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2508_06768_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# counts around the group sizes; displays of 1 to 4 warps' width, of few tiles
# (groups side by side) and of more
@pytest.mark.parametrize("wh", [(1, 9), (8, 33), (9, 40), (16, 70), (17, 31), (33, 64), (200, 900)])
@pytest.mark.parametrize("count", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 17, 31])
def test_images_of_a_call_are_independent(wh, count):
    import torch
    from paper_2508_06768_gb300.render import ScanConverter
    fan = I.Fan(21, 90, math.radians(75), 40.0)
    conv = ScanConverter(fan, *wh)
    rng = np.random.default_rng(count)
    x = torch.from_numpy(rng.standard_normal((count, 21, 90)).astype(np.float32)).cuda().requires_grad_(True)
    y = conv(x)
    g = torch.from_numpy(rng.standard_normal(tuple(y.shape)).astype(np.float32)).cuda()
    (gx,) = torch.autograd.grad(y, x, g)
    for c in range(count):
        xc = x[c].detach().clone().requires_grad_(True)
        yc = conv(xc)
        assert torch.equal(yc, y[c])
        assert torch.equal(torch.autograd.grad(yc, xc, g[c].clone())[0], gx[c])
    c = count - 1
    ref = oracle.scan_convert(x[c].detach().cpu().numpy().astype(np.float64), fan, conv.grid)
    refT = oracle.scan_convert_T(g[c].cpu().numpy().astype(np.float64), fan, 21, 90, conv.grid)
    assert np.abs(y[c].detach().cpu().numpy() - ref).max() <= 1e-5
    assert np.linalg.norm(gx[c].cpu().numpy() - refT) <= 1e-5 * max(np.linalg.norm(refT), 1e-30)


@pytest.mark.parametrize("wh", [(2100000, 1), (1, 2100000)])
def test_display_beyond_one_grid_of_tile_columns(wh):
    # 65625 columns of 32 pixels, of which one launch takes 65535
    import torch
    from paper_2508_06768_gb300.render import ScanConverter
    fan = I.Fan(9, 33, math.radians(75), 40.0)
    conv = ScanConverter(fan, *wh)
    x = torch.from_numpy(np.random.default_rng(1).standard_normal((9, 33)).astype(np.float32)).cuda()
    y = conv(x).cpu().numpy()
    ref = oracle.scan_convert(x.cpu().numpy().astype(np.float64), fan, conv.grid)
    assert np.abs(y - ref).max() <= 1e-5 and np.abs(ref).max() > 0
