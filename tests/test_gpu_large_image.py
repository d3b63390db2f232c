"""Images of more than 2,097,152 pixels (1,024 blocks of the prefix sum over the
pixels, beyond which their totals have a pass of their own), against the FP64
oracle, forward, backward and blending weights."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close
from tests.test_gpu_raster import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(2048, 1024), (2049, 1024), (1811, 1303)])
@pytest.mark.parametrize("F", [3, 4])
def test_image_around_the_limit(gpu, oracle, W, H, F):
    rng = np.random.default_rng(W)
    n = 60_000
    cam = scenes.make_camera((0.0, 0.0, 0.0), 900.0, 900.0, W / 2.0, H / 2.0, W, H)
    # half of the points everywhere, half on the last rows, where the offsets are largest
    u, z = rng.uniform(0, W, n), rng.uniform(1.0, 2.0, n)
    v = np.where(rng.random(n) < 0.5, rng.uniform(0, H, n), rng.uniform(H - 9, H, n))
    pos = np.stack([(u - W / 2.0) / 900.0 * z, (v - H / 2.0) / 900.0 * z, z], 1).astype(np.float32)
    op = rng.uniform(0.05, 0.9, n).astype(np.float32)
    feat = rng.normal(size=(n, F)).astype(np.float32)
    _compare(gpu, oracle, cam, pos, feat, op, head=False)
    opts = api.RasterOptions(n_channels=F)
    P, O, Fe = (torch.from_numpy(x).to(gpu) for x in (pos, op, feat))
    _, _, nc, ws = api.rasterize_fwd(cam, opts, P, Fe, O)
    b = api.point_weights(cam, opts, P, nc, ws)
    want = oracle.point_weights(cam, pos, feat, opacity=op)
    assert_cond_close(b.cpu().numpy(), want, want, what="b")
