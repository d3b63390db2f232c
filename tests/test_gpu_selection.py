"""Buckets of 257 to 1,024 fragments on an image with enough of them that a
warp selects the nearest fragments of each, with depths spread, in tied groups
and equal, and with blends shorter and longer than the selection, against the
FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close
from tests.test_gpu_raster import _compare, _product_widening

pytestmark = pytest.mark.gpu

SELECT_MIN = 4_096  # pixels from which warps select
W = H = 66


def _cloud(seed, pattern):
    rng = np.random.default_rng(seed)
    n = 358_000
    u, v, z = rng.uniform(-1, W + 1, n), rng.uniform(-1, H + 1, n), 1.0 + rng.random(n)
    lo, hi = 0.3, 0.95
    if pattern == "ties":  # a few fragments of a pixel at each of 64 depths
        z = 1.0 + np.floor(64 * rng.random(n)) / 64.0
    elif pattern == "clusters":  # most fragments at two depths: no threshold between the counts
        z = np.where(rng.random(n) < 0.9, 1.0 + 1e-6 * np.floor(2 * rng.random(n)), z)
    elif pattern == "equal":
        z = np.full(n, 1.5)
    elif pattern == "faint":  # the whole bucket blends
        lo, hi = 0.001, 0.01
    elif pattern == "long":  # about as many fragments blend as are selected
        lo, hi = 0.05, 0.6
    pos = np.stack([(u - W / 2.0) / 64.0 * z, (v - H / 2.0) / 64.0 * z, z], 1).astype(np.float32)
    cam = scenes.make_camera((0.0, 0.0, 0.0), 64.0, 64.0, W / 2.0, H / 2.0, W, H)
    return cam, pos, rng.uniform(lo, hi, n).astype(np.float32), rng


def _check_sizes(ref):
    m = ref["n_frags"]
    assert int(((m > 256) & (m <= 1024)).sum()) >= SELECT_MIN


PATTERNS = ("spread", "ties", "clusters", "equal", "faint", "long")


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("F", [3, 4, 8, 32, 64, 128])
def test_selection_matches_oracle(gpu, oracle, F, pattern):
    cam, pos, op, rng = _cloud(F, pattern)
    feat = rng.normal(size=(pos.shape[0], F)).astype(np.float32)
    _, ref = _compare(gpu, oracle, cam, pos, feat, op, head=False, with_bwd=F <= 8)
    _check_sizes(ref)


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("F", [32, 64, 128])
def test_selection_bf16_matches_oracle(gpu, oracle, F, pattern):
    cam, pos, op, rng = _cloud(100 + F, pattern)
    feat = torch.from_numpy(rng.normal(size=(pos.shape[0], F)).astype(np.float32)).to(torch.bfloat16)
    img, T, nc, _ = api.rasterize_fwd(cam, api.RasterOptions(n_channels=F, bf16=True), torch.from_numpy(pos).to(gpu),
                                      feat.to(gpu), torch.from_numpy(op).to(gpu))
    ref = oracle.raster_fwd(cam, pos, feat.float().numpy(), opacity=op, with_abs=True)
    _check_sizes(ref)
    ok = ref["flags"] == 0
    assert int((~ok).sum()) <= 2
    wp, _ = _product_widening(oracle, cam, pos, ref["n_contrib"])
    assert np.array_equal(nc.cpu().numpy()[ok], ref["n_contrib"][ok])
    assert_cond_close(T.cpu().numpy(), ref["T_final"], ref["T_final"] * wp, mask=ok, what="T_final")
    # the sums are the FP32 path's; the image is rounded to BF16 once (8 significant bits: 2^-8)
    got, want = img.float().cpu().numpy().astype(np.float64), ref["image"]
    bound = 1e-5 * ref["abs"] * wp[..., None] + np.abs(want) * 2.0 ** -8 * (1 + 1e-3)
    assert (np.abs(got - want) <= bound)[ok].all()
