"""The tile-sort binning at the lengths and depth distributions where its paths change: keys, order, ranges and
pair slots equal the oracle's."""
import numpy as np
import pytest

import oracle
from scenes import make_scene
from scenes.generate import camera_array

from gpu_common import gpu_render, read_discrete

pytestmark = pytest.mark.gpu


def _check(params, cams, W, H, cap):
    r, _, _, _ = gpu_render(params, cams, W, H, cap=cap)
    d = read_discrete(r)
    L = oracle.forward(params, cams, W, H)["lists"]
    assert d["status"] == 0 and d["total_pairs"] == len(L.keys)
    np.testing.assert_array_equal(d["keys"], L.keys)
    np.testing.assert_array_equal(d["vals"], L.vals)
    np.testing.assert_array_equal(d["ranges"], L.ranges)
    slots = d["slots"].astype(np.int64)
    assert np.array_equal(np.sort(slots), np.arange(len(slots)))
    first = d["offset"].astype(np.int64)[d["item"]]
    assert np.all((slots >= first) & (slots < first + d["count"].astype(np.int64)[d["item"]]))
    return r


def _heap(n, depth, seed=3):
    """n small Gaussians that all meet the tile at the image centre, at the given depths."""
    rng = np.random.default_rng(seed)
    W, H, f = 208, 192, 100.0
    uv = rng.uniform(-5.0, 5.0, (n, 2)) + 8.0
    z = depth(rng, n).astype(np.float32)
    means = np.concatenate([uv * z[:, None] / f, z[:, None]], 1).astype(np.float32)
    scales = np.full((n, 3), np.log(0.01), np.float32)
    quats = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1))
    logits = rng.normal(-3.0, 0.3, n).astype(np.float32)
    rgb = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    cam = camera_array(f, f, W / 2, H / 2, np.eye(3), np.zeros(3))
    return (means, scales, quats, logits, rgb), cam, W, H


DEPTHS = {
    "spread": lambda rng, n: rng.uniform(2.0, 6.0, n),
    "equal": lambda rng, n: np.full(n, 4.0),
    # most depths within a few hundred representable values, the rest far away
    "cluster": lambda rng, n: np.where(rng.random(n) < 0.9, 4.0 + rng.integers(0, 300, n) * 4.8e-7, rng.uniform(0.5, 9.0, n)),
}


@pytest.mark.parametrize("depths", sorted(DEPTHS))
@pytest.mark.parametrize("n", [1, 257, 2048, 2049, 4608, 4609, 12000])
def test_list_lengths(n, depths):
    """One long list (and its neighbours): the shortest, both sides of the longest list of a short-list
    block and of the longest list sorted in one piece, and one cut into pieces."""
    params, cam, W, H = _heap(n, DEPTHS[depths])
    r = _check(params, cam, W, H, cap=1 << 17)
    assert r.layout.bin_sort_launches == 4


@pytest.mark.parametrize("W,H,K,n", [(19 * 16, 8 * 16, 1, 900), (150 * 16 + 1, 16, 1, 500), (200, 150, 5, 1003),
                                     (640, 33, 3, 4100)])
def test_grids_and_views(W, H, K, n):
    """Just 152 tiles, one row of tiles, view boundaries inside projection blocks, ragged sizes."""
    s = make_scene("window500k", n=n, K=K, W=W, H=H, f=0.8 * min(W, 320))
    _check(s.params(), s.cams, W, H, cap=1 << 18)


@pytest.mark.parametrize("W,H,K,n", [(200, 150, 12, 40), (200, 150, 9, 1), (64, 48, 12, 40)])
def test_many_views_in_a_projection_block(W, H, K, n):
    """So few Gaussians that a projection block spans more views than it keeps cameras of in shared
    memory; the last one has too few tiles for the tile-sort binning."""
    s = make_scene("window500k", n=n, K=K, W=W, H=H, f=0.8 * W)
    _check(s.params(), s.cams, W, H, cap=1 << 16)
