"""Buckets whose fragments share their depths (the point index orders them) at
the sizes that one warp blends whole, for every narrow width, against the FP64
oracle."""
import numpy as np
import pytest

from paper_2403_16862_gb300 import scenes
from tests.test_gpu_raster import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [4, 8, 12, 24, 40])
@pytest.mark.parametrize("depths", ["equal", "few", "pairs", "wide"])
def test_tied_depths(gpu, oracle, F, depths):
    rng = np.random.default_rng(F)
    sizes = [9, 17, 31, 32, 33, 63, 64, 65, 97, 127, 128, 129, 190, 255, 256]
    W, H = 3 * len(sizes) + 3, 4
    cam = scenes.make_camera((0.0, 0.0, 0.0), 64.0, 64.0, W / 2.0, H / 2.0, W, H)
    pos = []
    for i, m in enumerate(sizes):
        if depths == "equal":
            z = np.full(m, 1.5)
        elif depths == "few":
            z = 1.0 + np.floor(3 * rng.random(m)) / 4
        elif depths == "pairs":
            z = 1.0 + np.repeat(rng.random(m // 2 + 1), 2)[:m]
        else:  # a span of more than 2^24 FP32 values
            z = np.where(np.arange(m) % 2 == 0, 0.2 + 0.01 * rng.random(m), 20.0 + rng.random(m))
        u, v = 3 * i + 2.0 + 0.3 * rng.random(m), 2.0 + 0.3 * rng.random(m)
        pos.append(np.stack([(u - W / 2.0) / 64.0 * z, (v - H / 2.0) / 64.0 * z, z], 1))
    pos = np.concatenate(pos).astype(np.float32)
    pos = pos[rng.permutation(len(pos))]
    op = rng.uniform(0.02, 0.3, len(pos)).astype(np.float32)
    feat = rng.normal(size=(len(pos), F)).astype(np.float32)
    _compare(gpu, oracle, cam, pos, feat, op, head=False)
