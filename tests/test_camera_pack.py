"""``native.cameras`` writes a camera in one piece; the fields equal those of a
write per field, also for values that only ctypes converts (too large for
float32 or int32)."""
import ctypes

import numpy as np
import pytest

from paper_2603_27151_gb300 import inputs as I
from paper_2603_27151_gb300 import native as N


@pytest.mark.parametrize("change", [{}, dict(fx=1e39), dict(near=-1e300), dict(width=2 ** 33 + 5), dict(cx=float("nan")),
                                    dict(cy=1e-45), dict(R=np.arange(9.0).reshape(3, 3) / 7), dict(t=[1, 2.5, -3])])
def test_fields_equal_those_written_one_by_one(change):
    cams = [I.look_at([0.3, 0.2, 3.0], 64, 48), I.look_at([1.0, -0.2, 2.0], 31, 77), I.look_at([0.0, 2.2, 1.0], 1, 1)]
    for k, v in change.items():
        setattr(cams[1], k, v)
    assert N._CAMERA.size == ctypes.sizeof(N.ds_camera)
    assert bytes(N.cameras(cams)) == bytes(N._cameras_by_field(cams))
    assert len(N.cameras([])) == 0
