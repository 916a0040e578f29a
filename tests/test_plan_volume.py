"""A batch call on a volume that its plan's fans do not fit."""
import ctypes as C
import math

import torch

from paper_2508_06768_gb300 import binding as B
from paper_2508_06768_gb300 import inputs as I


def test_plan_on_a_much_finer_volume_is_refused():
    # positions are fixed point and a ray may span 2^29 voxels: the plan checks
    # it for its own spacing, the call has to for the one it is given
    vol = torch.zeros((16, 16, 16))
    prm, fans = I.Params(seed=1, mode=1), [I.Fan(8, 64, math.radians(40), 30.0), I.Fan(3, 9, 0.5, 3.0)]
    plan, _, _, wsb = B.batch_plan(vol, (1.0,) * 3, (0.0,) * 3, fans, prm)
    pd, vp = B.params_desc(prm), C.c_void_p

    def call(spacing, ws_bytes):
        vd = B.volume_desc(vol, spacing, (0.0,) * 3)
        return B.load().diffus_render_batch(vp(256), C.byref(vd), vp(256), vp(plan.data_ptr()), vp(256), C.byref(pd),
                                            vp(256), None, None, None, None, None, vp(256), ws_bytes, None, None)
    assert call((1.0, 1.0, 1e-8), 1 << 40) == -3
    assert call((1.0, 5e-324, 1.0), 1 << 40) == -3
    assert call((1.0, 1.0, 1e-7), 16) == -6        # 3e8 voxels: on to the next check
    assert call((1.0, 1.0, 1.0), 16) == -6
