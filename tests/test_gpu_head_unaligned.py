"""The SH head on rows that start between 16-byte boundaries, for widths of each
way the forward reads them, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [37, 40, 42, 64])
@pytest.mark.parametrize("n", [1, 33, 1_000])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_rows_at_an_odd_offset(gpu, oracle, F, n, dtype):
    rng = np.random.default_rng(1000 * F + n)
    cam = scenes.make_camera((0.3, -0.2, -2.0), 100.0, 100.0, 50.0, 40.0, 100, 80)
    pos = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    flat = torch.from_numpy(rng.normal(0, 0.5, n * F + 1).astype(np.float32)).to(dtype).to(gpu)
    h = flat[1:].view(n, F)
    assert h.data_ptr() % 4 == flat.element_size() % 4 and h.is_contiguous()
    hf = h.float().cpu().numpy()
    da, dc = rng.normal(size=n).astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32)
    P, A, C = (torch.from_numpy(x).to(gpu) for x in (pos, da, dc))
    alpha, color = api.sh_head_fwd(cam, P, h)
    dh = api.sh_head_bwd(cam, P, h, A, C)
    o_a, o_c, o_ab = oracle.sh_head_fwd(cam, pos, hf, with_abs=True)
    o_dh, o_dab = oracle.sh_head_bwd(cam, pos, hf, da, dc, with_abs=True)
    assert_cond_close(alpha.cpu().numpy(), o_a, o_a, what="alpha")
    assert_cond_close(color.cpu().numpy(), o_c, o_ab, what="color")
    assert_cond_close(dh.cpu().numpy(), o_dh, o_dab, what="dh")
