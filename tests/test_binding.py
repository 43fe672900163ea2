"""The Python binding's argument marshalling. CPU only."""
import numpy as np
import pytest


def test_camera_bytes_equal_the_fields():
    """The packed form of a camera is the struct that the fields give, for the number
    types that callers have, and for what it hands to the field-by-field form."""
    from types import SimpleNamespace
    from paper_2603_15186_gb300 import camera_array, camera_struct, renderer
    R = np.arange(9, dtype=np.float64).reshape(3, 3)
    base = dict(pos=[1, 2.5, 3], R_wc=R, fx=100, fy=np.float32(90.5), cx=32.0, cy=np.float64(24), width=64,
                height=np.int64(48), tau=2)
    cams = [SimpleNamespace(**{**base, **d}) for d in (
        {}, {"pos": np.float32([4, 5, 6]), "R_wc": R.T}, {"R_wc": R.reshape(9).tolist()}, {"width": 64.0},
        {"tau": np.array(3.5)}, {"fx": float("inf")}, {"fx": 1e39}, {"pos": np.float32([[7, 8, 9]])})]
    want = [bytes(renderer._camera_by_field(c)) for c in cams]
    assert [bytes(camera_struct(c)) for c in cams] == want
    assert bytes(camera_array(cams)) == b"".join(want) and len(camera_array([])) == 0
    for bad in ({"pos": [1, 2]}, {"R_wc": R[:2]}, {"width": None}):
        with pytest.raises((TypeError, ValueError)):
            camera_array([SimpleNamespace(**{**base, **bad})])
