"""Forward and backward of buckets whose sizes lie at the edges of the blend
paths (lane groups, one warp, selection by one warp, CTA), with depths spread,
clustered and equal, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 3, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 255, 256, 257, 300, 1023, 1024, 1025, 2049)


def _columns(seed, F, alpha_lo, alpha_hi):
    """One bucket of every size and depth pattern: points behind the centers
    of pixels three apart."""
    rng = np.random.default_rng(seed)
    W, H = 3 * len(SIZES) + 3, 12
    cam = scenes.make_camera((0.0, 0.0, 0.0), 64.0, 64.0, W / 2.0, H / 2.0, W, H)
    pos = []
    for j in range(3):
        for i, m in enumerate(SIZES):
            z = 1.0 + rng.random(m)
            if j == 1:  # most fragments in one tight cluster in front
                z = np.where(rng.random(m) < 0.9, 1.0 + 1e-6 * np.floor(rng.random(m) * 8), z)
            if j == 2:  # equal depths: the point index decides
                z = np.full(m, 1.5)
            u, v = 3 * i + 2.0 + 0.3 * rng.random(m), 4 * j + 2.0 + 0.3 * rng.random(m)
            pos.append(np.stack([(u - W / 2.0) / 64.0 * z, (v - H / 2.0) / 64.0 * z, z], 1))
    pos = np.concatenate(pos).astype(np.float32)
    n = pos.shape[0]
    perm = rng.permutation(n)
    return cam, pos[perm], rng.uniform(alpha_lo, alpha_hi, n).astype(np.float32), \
        rng.normal(size=(n, F)).astype(np.float32), rng.normal(size=(H, W, F)).astype(np.float32)


@pytest.mark.parametrize("F", [3, 4, 8, 12, 32, 64, 128])
@pytest.mark.parametrize("alpha", [(0.05, 0.6), (0.001, 0.01)])
def test_bucket_sizes_match_oracle(gpu, oracle, F, alpha):
    cam, pos, op, feat, g = _columns(F, F, *alpha)
    ref = oracle.raster_fwd(cam, pos, feat, op, with_abs=True)
    rb = oracle.raster_bwd(cam, pos, feat, g, op, with_abs=True)
    P, O, Fe, G = (torch.from_numpy(x).to(gpu) for x in (pos, op, feat, g))
    opts = api.RasterOptions(n_channels=F)
    img, T, nc, ws = api.rasterize_fwd(cam, opts, P, Fe, O)
    d_op, d_feat = api.rasterize_bwd(cam, opts, P, Fe, O, T, nc, G, ws)
    ok = ref["flags"] == 0
    assert ok.mean() > 0.99
    assert np.array_equal(nc.cpu().numpy()[ok], ref["n_contrib"][ok])
    # a blend of n fragments rounds its transmittance n times
    rtol = max(1e-5, float(ref["n_contrib"].max()) * 2.0 ** -24)
    assert_cond_close(img.cpu().numpy(), ref["image"], ref["abs"], rtol=rtol, mask=ok[..., None], what="image")
    if ok.all():
        assert_cond_close(d_feat.cpu().numpy(), rb["d_feat"], rb["abs_feat"], rtol=rtol, what="d_feat")
        assert_cond_close(d_op.cpu().numpy(), rb["d_opacity"], rb["abs_opacity"], rtol=rtol, what="d_opacity")
