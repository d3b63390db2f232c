"""The binning of fragments into pixel buckets: chunk edges, clouds whose
chunks reach over many windows of counters (unordered), clouds in one pixel
and off-image corners, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,layout", [(1, "uniform"), (255, "uniform"), (257, "pixel"), (1_023, "border"),
                                      (5_000, "uniform"), (320_001, "uniform"), (320_001, "grouped"),
                                      (1_900_001, "uniform"), (1_900_001, "grouped")])
def test_binned_fragments_match_oracle(gpu, oracle, n, layout):
    rng = np.random.default_rng(n)
    W, H, F = 331, 203, 4
    cam = scenes.make_camera((0.0, 0.0, 0.0), 200.0, 200.0, W / 2.0, H / 2.0, W, H)
    u, v = rng.uniform(-3, W + 3, n), rng.uniform(-3, H + 3, n)
    if layout == "pixel":
        u, v = np.full(n, 70.2), np.full(n, 100.9)
    elif layout == "border":
        u = np.where(rng.random(n) < 0.5, rng.uniform(-0.6, 0.6, n), W + rng.uniform(-0.6, 0.6, n))
    elif layout == "grouped":  # runs of 64 points on a few pixels, the runs anywhere
        k = np.arange(n) // 64
        u, v = (c[k] + rng.uniform(0, 9, n) for c in (u, v))
    z = rng.uniform(1.0, 2.0, n)
    pos = np.stack([(u - W / 2.0) / 200.0 * z, (v - H / 2.0) / 200.0 * z, z], 1).astype(np.float32)
    op = rng.uniform(0.05, 0.95, n).astype(np.float32)
    feat = rng.normal(size=(n, F)).astype(np.float32)
    ref = oracle.raster_fwd(cam, pos, feat, op, with_abs=True)
    img, T, nc, _ = api.rasterize_fwd(cam, api.RasterOptions(n_channels=F), *(torch.from_numpy(x).to(gpu)
                                                                             for x in (pos, feat, op)))
    ok = ref["flags"] == 0
    assert ok.mean() > 0.999
    assert np.array_equal(nc.cpu().numpy()[ok], ref["n_contrib"][ok])
    rtol = max(1e-5, float(ref["n_contrib"].max()) * 2.0 ** -24)
    assert_cond_close(img.cpu().numpy(), ref["image"], ref["abs"], rtol=rtol, mask=ok[..., None], what="image")
