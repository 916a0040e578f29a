"""What render() takes for its plain arguments: the packed form of the native
node reads the same values as the C descriptors of the Python function, and
refuses what they refuse."""
import ctypes as C
import math

import numpy as np
import pytest

from paper_2508_06768_gb300 import binding as B
from paper_2508_06768_gb300 import inputs as I

FAN = I.Fan(7, 90, math.radians(50), 33.0, 5.0, 0.5)


def _descs(spacing, origin, fan, prm, ctr):
    """The bytes of the same call through the ctypes descriptors."""
    six = (C.c_double * 6)(*[float(spacing[i]) for i in range(3)], *[float(origin[i]) for i in range(3)])
    return bytes(six) + bytes(B.fan_desc(fan)) + bytes(B.params_desc(prm, ctr))


@pytest.mark.parametrize("spacing,origin", [((1.0, 0.9, 1.1), (0.25, 0, -0.5)), ([1, 2, 3], np.zeros(3)),
                                            (np.array([0.5, 0.5, 0.5, 9.0]), (1.0, 2.0, 3.0, 4.0))])
def test_packed_call_holds_the_descriptors(spacing, origin):
    prm = I.Params(seed=2**63 + 5, mode=1, atten=1)
    assert B.pack_call(spacing, origin, FAN, prm, 2**32 + 3) == _descs(spacing, origin, FAN, prm, 2**32 + 3)


@pytest.mark.parametrize("spacing,origin", [((1.0, 1.0, 1.0, 0.5), (0.0, 0.0)), ((1.0, 1.0), (0.0,) * 4),
                                            ((1.0,) * 6, ()), ((1.0,) * 5, (0.0,))])
def test_short_spacing_or_origin_is_refused(spacing, origin):
    # not made up from the other one's numbers
    with pytest.raises(IndexError):
        _descs(spacing, origin, FAN, I.Params(seed=1), 0)
    with pytest.raises(IndexError):
        B.pack_call(spacing, origin, FAN, I.Params(seed=1))
