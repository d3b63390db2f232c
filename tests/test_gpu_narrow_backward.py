"""The backward of narrow widths on images with enough pixels of a few blended
fragments that lane groups take them, against the FP64 oracle."""
import numpy as np
import pytest

from paper_2403_16862_gb300 import scenes
from tests.test_gpu_raster import _compare

pytestmark = pytest.mark.gpu

GROUP_MIN = 32_768  # pixels from which the lists go to lane groups


@pytest.mark.parametrize("F,per_pixel,lo,hi", [(4, 5.0, 3, 8), (8, 6.5, 5, 8), (12, 12.0, 9, 16), (16, 12.0, 9, 16),
                                               (24, 20.0, 17, 64), (4, 14.0, 9, 256)])
def test_long_lists_of_short_blends(gpu, oracle, F, per_pixel, lo, hi):
    rng = np.random.default_rng(int(10 * per_pixel) + F)
    W, H = 317, 241
    n = int(per_pixel / 4 * W * H)
    cam = scenes.make_camera((0.0, 0.0, 0.0), 300.0, 300.0, W / 2.0, H / 2.0, W, H)
    u, v, z = rng.uniform(0, W, n), rng.uniform(0, H, n), rng.uniform(1.0, 2.0, n)
    pos = np.stack([(u - W / 2.0) / 300.0 * z, (v - H / 2.0) / 300.0 * z, z], 1).astype(np.float32)
    op = rng.uniform(0.02, 0.4, n).astype(np.float32)
    feat = rng.normal(size=(n, F)).astype(np.float32)
    _, ref = _compare(gpu, oracle, cam, pos, feat, op, head=False)
    assert int(((ref["n_contrib"] >= lo) & (ref["n_contrib"] <= hi)).sum()) >= GROUP_MIN
