"""The stand-alone grid adjoint (inpc_query_hashgrid_bwd) at the edges of its
dispatch (levels per warp pair, level groups for tables beyond L2) and of its
point chunks, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from tests._parity import assert_cond_close
from paper_2403_16862_gb300 import api, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,log2_T,n,grouped", [
    (1, 10, 1, False), (4, 12, 777, False), (5, 12, 17, True), (8, 14, 4097, True), (9, 14, 389, False),
    (16, 16, 1, False), (16, 16, 40_009, True), (16, 21, 6_001, True), (17, 12, 1_283, False), (32, 21, 2_003, True),
])
def test_adjoint_matches_oracle(gpu, oracle, levels, log2_T, n, grouped):
    res = scenes.geometric_resolutions(levels, 16, 4096)
    rng = np.random.default_rng(levels * 1000 + n)
    pos = rng.random((n, 3)).astype(np.float32)
    if grouped:  # runs of points that share coarse cells, then jump
        pos = (np.repeat(rng.random((n // 50 + 1, 3)), 50, 0)[:n] * 0.97 + 0.03 * pos).astype(np.float32)
    pos[0] = (1.0, 0.0, 1.0)  # the grid's corner
    dh = rng.normal(size=(n, 4 * levels)).astype(np.float32)
    dh[rng.random(n) < 0.1] = 0.0
    ref, ab = oracle.hash_bwd(res, log2_T, 4, pos, dh, with_abs=True)
    desc = api.hashgrid_desc(res, log2_T)
    grad = torch.ones(ref.shape, dtype=torch.float32, device=gpu)
    api.query_hashgrid_bwd(desc, torch.from_numpy(pos).to(gpu), torch.from_numpy(dh).to(gpu), grad)
    # accumulates onto what the table gradient holds (here ones)
    assert_cond_close(grad.cpu().numpy(), ref + 1.0, ab + 1.0, what="table gradient")
