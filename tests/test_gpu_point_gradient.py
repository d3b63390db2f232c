"""Gradients of point counts around those from which a warp takes more points,
against the FP64 oracle."""
import numpy as np
import pytest

from paper_2403_16862_gb300 import scenes
from tests.test_gpu_raster import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [6, 32, 64, 128])
@pytest.mark.parametrize("n", [1, 7, 4_865, 19_457, 38_911, 77_825])
def test_gradients_across_points_per_warp(gpu, oracle, F, n):
    rng = np.random.default_rng(n + F)
    W, H = 211, 133
    cam = scenes.make_camera((0.0, 0.0, 0.0), 200.0, 200.0, W / 2.0, H / 2.0, W, H)
    u, v, z = rng.uniform(-2, W + 2, n), rng.uniform(-2, H + 2, n), rng.uniform(1.0, 2.0, n)
    pos = np.stack([(u - W / 2.0) / 200.0 * z, (v - H / 2.0) / 200.0 * z, z], 1).astype(np.float32)
    op = rng.uniform(0.05, 0.6, n).astype(np.float32)
    feat = rng.normal(0, 0.5, (n, F)).astype(np.float32)
    _compare(gpu, oracle, cam, pos, feat, op, head=False)
    _compare(gpu, oracle, cam, pos, feat, None, head=True)
