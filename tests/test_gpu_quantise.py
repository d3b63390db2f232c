"""Leaf draws where the weights' quantisation is decided close to a rounding
boundary, and for maxima at the ends of the FP64 range, bit-exact against the
oracle."""
import numpy as np
import pytest
import torch

from paper_2403_16862_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def _tree(w):
    L = w.shape[0]
    g = int(np.ceil(L ** (1 / 3)))
    ijk = np.stack(np.unravel_index(np.arange(L), (g, g, g)), 1)
    return scenes.Octree(centers=((ijk + 0.5) / 16.0).astype(np.float32), levels=np.full(L, 4, np.int32),
                         weights=w.astype(np.float64), root_size=1.0)


@pytest.mark.parametrize("scale", [1.0, 3.0, 1e-305, 1e-290, 1e290, 7e307])
def test_draws_at_rounding_boundaries(gpu, oracle, scale):
    rng = np.random.default_rng(1)
    L = 4099  # beyond one scan block
    k = rng.integers(0, 1 << 29, L).astype(np.float64)
    k[: L // 2] = rng.integers(0, 64, L // 2)
    half = (k + 0.5) / 2.0 ** 29
    w = half * (1.0 + rng.integers(-3, 4, L) * 2.0 ** -52)  # at and next to half-integers
    w[::7] = k[::7] / 2.0 ** 29
    w[5], w[6], w[11] = 0.0, -0.0, 1.0
    tree = _tree(np.minimum(w, 1.0) * scale)
    n = 50_000
    c, l, ww = (torch.from_numpy(x).to(gpu) for x in (tree.centers, tree.levels, tree.weights))
    leaf, pos, counts = api.sample_octree(c, l, ww, 1.0, 9, 2, n, with_counts=True)
    o_leaf, o_pos, o_counts = oracle.sample_octree(tree, 9, 2, n)
    assert np.array_equal(leaf.cpu().numpy(), o_leaf)
    assert np.array_equal(pos.cpu().numpy(), o_pos.astype(np.float32))
    assert np.array_equal(counts.cpu().numpy(), o_counts)


@pytest.mark.parametrize("n", [1, 2_047, 2_049, 70_001])
@pytest.mark.parametrize("rounds", [0, 1, 5])
def test_view_samples_at_tile_edges(gpu, oracle, n, rounds):
    tree = scenes.make_octree(3, 4096)
    cam = scenes.look_at_camera((0.5, 0.4, -0.8), (0.6, 0.5, 0.5), 90.0, 90.0, 32.0, 24.0, 64, 48)
    c, l, p = (torch.from_numpy(x).to(gpu) for x in (tree.centers, tree.levels, tree.weights))
    w = api.view_weights(c, l, p, 1.0, cam)
    o_w = oracle.view_weights(tree, cam)
    assert np.array_equal(w.cpu().numpy(), o_w)
    leaf, pos, left = api.sample_octree_view(c, l, w, 1.0, cam, 4, 1, n, max_rounds=rounds)
    o_leaf, o_pos, o_left = oracle.sample_view(tree, o_w, cam, 4, 1, n, max_rounds=rounds)
    assert np.array_equal(leaf.cpu().numpy(), o_leaf)
    assert np.array_equal(pos.cpu().numpy(), o_pos.astype(np.float32))
    assert int(left) == o_left
