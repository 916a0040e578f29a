"""The HU map's lookup table at the sizes real calibrations give it: more entries
than a block has threads, more bytes than a kernel's shared memory holds without
asking, and the largest table before the search takes over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("lo,hi,n", [(-1024, 3071, 5_000_000),       # 4096 entries, 16 KB
                                     (-6000, 6300, 15_100_000),      # 12301 entries: just over 48 KB
                                     (-12288, 12287, 30_000_000),    # 24576 entries: the largest table
                                     (-12288, 12288, 30_000_000)])   # one more: the search
def test_hu_table_of_many_entries(lo, hi, n, bf16):
    import torch
    from paper_2508_06768_gb300 import binding as B
    pts = [float(lo), lo // 2 + 0.25, lo // 8 - 0.5, 0.75, float(hi // 2), float(hi)]
    z = [0.1, 1.2, 1.45, 1.5, 3.0, 7.8]
    dt = torch.bfloat16 if bf16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n)
    hu = torch.randint(max(lo - 200, -32768), min(hi + 200, 32767) + 1, (n,), device="cuda", generator=g,
                       dtype=torch.int32).to(torch.int16)
    hu[:hi - lo + 1] = torch.arange(lo, hi + 1, device="cuda", dtype=torch.int32).to(torch.int16)   # every entry
    full = B.hu_to_z(hu, pts, z, dtype=dt)
    # parts too small for a table of this size are searched
    step = -(-n // 3 // 8) * 8
    parts = torch.cat([B.hu_to_z(hu[i:i + step].clone(), pts, z, dtype=dt) for i in range(0, n, step)])
    assert torch.equal(full, parts)
    m = hi - lo + 1000
    ref = np.interp(hu[:m].cpu().numpy().astype(np.float64), pts, z)
    tol = 2.0 ** -8 if bf16 else 3e-7
    assert np.all(np.abs(full[:m].float().cpu().numpy() - ref) <= np.abs(ref) * tol * 1.01)
