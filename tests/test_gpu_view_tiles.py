"""View-specific samples at the sizes where the tiles of slots change, with a
view that few leaves lie in, so that most slots go through every round;
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rounds", [(257, 3), (155_648, 2), (155_649, 2), (400_003, 1), (1_300_003, 2)])
def test_slots_across_tiles(gpu, oracle, n, rounds):
    tree = scenes.make_octree(3, 4096)
    cam = scenes.look_at_camera((0.5, 0.5, 0.5), (0.6, 0.5, 0.7), 90.0, 90.0, 32.0, 24.0, 64, 48)
    c, l, w = (torch.from_numpy(x).to(gpu) for x in (tree.centers, tree.levels, tree.weights))
    leaf, pos, left = api.sample_octree_view(c, l, w, 1.0, cam, 4, 1, n, max_rounds=rounds)
    o_leaf, o_pos, o_left = oracle.sample_view(tree, tree.weights, cam, 4, 1, n, max_rounds=rounds)
    assert o_left > n // 2
    assert np.array_equal(leaf.cpu().numpy(), o_leaf)
    assert np.array_equal(pos.cpu().numpy(), o_pos.astype(np.float32))
    assert int(left) == o_left
