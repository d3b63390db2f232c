"""Rasterizer buffers at the smallest alignment the entry points accept (4
bytes where the channel count is not a multiple of 4), with empty pixels,
against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu


def _offset(gpu, shape, fill):
    """A contiguous FP32 tensor that starts 4 bytes behind a 512-byte boundary."""
    t = torch.full((int(np.prod(shape)) + 1,), fill, device=gpu)[1:].view(shape)
    assert t.data_ptr() % 8 == 4
    return t


@pytest.mark.parametrize("F", [2, 3, 6, 10, 30])
def test_image_at_a_four_byte_offset(gpu, oracle, F):
    rng = np.random.default_rng(F)
    W, H, n = 45, 31, 300
    cam = scenes.make_camera((0.0, 0.0, 0.0), 40.0, 40.0, W / 2.0, H / 2.0, W, H)
    z = rng.uniform(1.0, 2.0, n)
    # one half of the image stays empty
    u, v = rng.uniform(0, W / 2.0, n), rng.uniform(0, H, n)
    pos = np.stack([(u - W / 2.0) / 40.0 * z, (v - H / 2.0) / 40.0 * z, z], 1).astype(np.float32)
    op = rng.uniform(0.05, 0.95, n).astype(np.float32)
    feat = rng.normal(size=(n, F)).astype(np.float32)
    g = rng.normal(size=(H, W, F)).astype(np.float32)
    ref = oracle.raster_fwd(cam, pos, feat, op, with_abs=True)
    rb = oracle.raster_bwd(cam, pos, feat, g, op, with_abs=True)
    assert (ref["n_frags"] == 0).any() and (ref["flags"] == 0).all()
    opts = api.RasterOptions(n_channels=F)
    P, O = torch.from_numpy(pos).to(gpu), torch.from_numpy(op).to(gpu)
    feat_t, g_t = _offset(gpu, (n, F), 0.0), _offset(gpu, (H, W, F), 0.0)
    feat_t.copy_(torch.from_numpy(feat))
    g_t.copy_(torch.from_numpy(g))
    nan = float("nan")
    out = (_offset(gpu, (H, W, F), nan), torch.full((H, W), nan, device=gpu),
           torch.full((H, W), -1, dtype=torch.int32, device=gpu))
    img, T, nc, ws = api.rasterize_fwd(cam, opts, P, feat_t, O, out=out)
    d_op, d_feat = api.rasterize_bwd(cam, opts, P, feat_t, O, T, nc, g_t, ws,
                                     out=(torch.empty(n, device=gpu), _offset(gpu, (n, F), nan)))
    assert np.array_equal(nc.cpu().numpy(), ref["n_contrib"])
    assert_cond_close(img.cpu().numpy(), ref["image"], ref["abs"], what="image")
    assert_cond_close(T.cpu().numpy(), ref["T_final"], ref["T_final"], what="T_final")
    assert_cond_close(d_feat.cpu().numpy(), rb["d_feat"], rb["abs_feat"], what="d_feat")
    assert_cond_close(d_op.cpu().numpy(), rb["d_opacity"], rb["abs_opacity"], what="d_opacity")
