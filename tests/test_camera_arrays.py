"""The camera struct from every kind of array that a camera may hold (no GPU)."""
import types

import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api

R = np.array([[0.36, 0.48, -0.8], [-0.8, 0.6, 0.0], [0.48, 0.64, 0.6]])
T = np.array([0.1, -2.0, 3.5])


def _masked(x):
    return np.ma.masked_array(x.astype(np.float32), mask=np.zeros(x.shape, bool))


KINDS = {
    "float32": lambda x: x.astype(np.float32),
    "float64": lambda x: x,
    "list": lambda x: x.tolist(),
    "tensor": lambda x: torch.from_numpy(x),
    "float32 tensor": lambda x: torch.from_numpy(x).float(),
    "matrix": lambda x: np.matrix(x.astype(np.float32)),
    "masked": _masked,
    "strided": lambda x: np.repeat(x.astype(np.float32), 2, axis=-1)[..., ::2],
    "fortran": lambda x: np.asfortranarray(x.astype(np.float32)),
    "flat": lambda x: x.astype(np.float32).ravel(),
    "column": lambda x: x.astype(np.float32).reshape(-1, 1),
    "read-only": lambda x: np.frombuffer(x.astype(np.float32).tobytes(), np.float32).reshape(x.shape),
}


@pytest.mark.filterwarnings("ignore")
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_camera_of(kind):
    cam = types.SimpleNamespace(R=KINDS[kind](R), t=KINDS[kind](T), fx=2.0, fy=3.0, cx=4.0, cy=5.0, width=6, height=7,
                                near=0.1, far=9.0)
    c = api.camera(cam)
    assert list(c.R) == R.astype(np.float32).ravel().tolist()
    assert list(c.t) == T.astype(np.float32).tolist()


@pytest.mark.parametrize("bad", [np.zeros((2, 3), np.float32), np.zeros(10, np.float32), [0.0] * 8])
def test_wrong_sizes_are_refused(bad):
    cam = types.SimpleNamespace(R=bad, t=T, fx=1, fy=1, cx=1, cy=1, width=6, height=7, near=0.1, far=9.0)
    with pytest.raises(RuntimeError):
        api.camera(cam)
