"""Per-point blending weights of pixels whose blends lie at the edges of the
ways they are walked (8 lanes, a warp, several chunks), against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 65, 200)


@pytest.mark.parametrize("width", [len(SIZES) * 3 + 3, 1_500])
@pytest.mark.parametrize("alpha", [(0.05, 0.6), (0.001, 0.01)])
def test_columns(gpu, oracle, width, alpha):
    rng = np.random.default_rng(width)
    W, H = width, 40
    cam = scenes.make_camera((0.0, 0.0, 0.0), 64.0, 64.0, W / 2.0, H / 2.0, W, H)
    pos = []
    for j in range(12):
        for i, m in enumerate(SIZES):
            z = 1.0 + rng.random(m)
            u, v = 3 * ((i + 5 * j) % len(SIZES)) + 2.0 + 0.3 * rng.random(m), 3 * j + 2.0 + 0.3 * rng.random(m)
            pos.append(np.stack([(u - W / 2.0) / 64.0 * z, (v - H / 2.0) / 64.0 * z, z], 1))
    pos = np.concatenate(pos).astype(np.float32)
    pos = pos[rng.permutation(len(pos))]
    op = rng.uniform(*alpha, len(pos)).astype(np.float32)
    feat = np.ones((len(pos), 64), np.float32)
    ref = oracle.raster_fwd(cam, pos, feat[:, :1], op)
    want = oracle.point_weights(cam, pos, feat[:, :1], opacity=op)
    assert (ref["flags"] == 0).all()
    opts = api.RasterOptions(n_channels=64)
    P, O, Fe = (torch.from_numpy(x).to(gpu) for x in (pos, op, feat))
    img, T, nc, ws = api.rasterize_fwd(cam, opts, P, Fe, O)
    b = api.point_weights(cam, opts, P, nc, ws)
    assert np.array_equal(nc.cpu().numpy(), ref["n_contrib"])
    # a blend of n fragments rounds its transmittance n times; every term is non-negative
    rtol = max(1e-5, float(ref["n_contrib"].max()) * 2.0 ** -24)
    assert_cond_close(b.cpu().numpy(), want, want, rtol=rtol, what="b")
