"""gs.camera over every form of R and t, and the pose delta of zero, against
the general formula."""
import math

import numpy as np
import pytest
import torch

from paper_2510_06644_gb300 import gs
from paper_2510_06644_gb300.autograd import apply_pose_delta

R = np.array([[0.36, 0.48, -0.8], [-0.8, 0.6, 0.0], [0.48, 0.64, 0.6]])
T = np.array([0.1, -0.2, 0.3])


def _cam(R, t):
    return {"R": R, "t": t, "fx": 50.0, "fy": 51.0, "cx": 31.5, "cy": 23.5, "W": 64, "H": 48}


@pytest.mark.parametrize("form", ["f64", "f32", "flat", "strided", "swapped", "list", "tensor"])
def test_camera_forms(form):
    make = {"f64": lambda a: a.copy(), "f32": lambda a: a.astype(np.float32), "flat": lambda a: a.reshape(-1).copy(),
            "strided": lambda a: np.stack([a, a], -1)[..., 0], "swapped": lambda a: np.asfortranarray(a),
            "list": lambda a: a.tolist(), "tensor": lambda a: torch.from_numpy(a.copy())}[form]
    c = gs.camera(_cam(make(R), make(T)))
    assert list(c.R) == R.astype(np.float32).reshape(9).tolist()
    assert list(c.t) == T.astype(np.float32).tolist()


def test_camera_refuses_wrong_sizes():
    with pytest.raises(RuntimeError):
        gs.camera(_cam(R[:2], T))
    with pytest.raises(RuntimeError):
        gs.camera(_cam(R, np.zeros(4)))


def test_zero_delta_is_the_limit():
    z = apply_pose_delta(_cam(R, T), np.zeros(6))
    assert np.array_equal(z["R"], R) and np.array_equal(z["t"], T) and z["W"] == 64
    z["R"][:] = 0  # a copy: the caller's camera stays
    assert R[0, 0] == 0.36
    # the smallest delta takes the matrices: the same pose within its own size
    s = apply_pose_delta(_cam(R, T), np.full(6, 1e-12))
    assert np.abs(s["R"] - R).max() < 4e-12 and np.abs(s["t"] - T).max() < 4e-12
    n = apply_pose_delta(_cam(np.full((3, 3), math.nan), T), np.zeros(6))
    assert np.isnan(n["R"]).all()
