"""The stand-alone grid adjoint on both sides of the number of points from
which the fine levels of a large table go level group by level group, against
the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes
from tests._parity import assert_cond_close

pytestmark = pytest.mark.gpu


# the fine levels (8 of 16, 16 of 32) stay in one launch up to 64 MB of touched sectors, the coarse ones up to 96 MB
# (all 8 of 12/20, five of 9/21, 10 of 24/21), all of them up to 112 MB
@pytest.mark.parametrize("levels,log2_T,n", [(16, 20, 32_768), (16, 20, 32_769), (16, 21, 40_001), (32, 20, 16_384),
                                             (32, 20, 16_385), (32, 20, 1), (12, 20, 120_001), (9, 21, 200_003),
                                             (24, 21, 90_001), (6, 21, 300_007), (20, 19, 70_001)])
def test_adjoint_around_the_split(gpu, oracle, levels, log2_T, n):
    res = scenes.geometric_resolutions(levels, 16, 4096)
    rng = np.random.default_rng(levels + n)
    pos = rng.random((n, 3)).astype(np.float32)
    dh = rng.normal(size=(n, 4 * levels)).astype(np.float32)
    ref, ab = oracle.hash_bwd(res, log2_T, 4, pos, dh, with_abs=True)
    grad = torch.zeros(ref.shape, dtype=torch.float32, device=gpu)
    api.query_hashgrid_bwd(api.hashgrid_desc(res, log2_T), torch.from_numpy(pos).to(gpu),
                           torch.from_numpy(dh).to(gpu), grad)
    assert_cond_close(grad.cpu().numpy(), ref, ab, what="table gradient")
