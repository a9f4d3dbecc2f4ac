"""One tile's list at exactly the lengths where the tile-sort binning changes its path, for several depth distributions:
keys, order, ranges and pair slots equal the oracle's."""
import numpy as np
import pytest

import oracle
from scenes.generate import camera_array

from tests.test_gpu_tile_sort import _check

W, H, F = 208, 192, 100.0  # 13 x 12 tiles


def heap(n, depth, seed=3):
    """n small Gaussians in the middle of tile (6, 6), none of which reaches another tile."""
    rng = np.random.default_rng(seed)
    uv = rng.uniform(-2.0, 2.0, (n, 2)) + [104 - W / 2, 104 - H / 2]
    z = depth(rng, n).astype(np.float32)
    means = np.concatenate([uv * z[:, None] / F, z[:, None]], 1).astype(np.float32)
    params = (means, np.full((n, 3), np.log(0.005), np.float32), np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)),
              rng.normal(-3.0, 0.3, n).astype(np.float32), rng.uniform(0, 1, (n, 3)).astype(np.float32))
    return params, camera_array(F, F, W / 2, H / 2, np.eye(3), np.zeros(3))


DEPTHS = {
    "spread": lambda rng, n: rng.uniform(2.0, 6.0, n),
    "equal": lambda rng, n: np.full(n, 4.0),
    # a wall seen through scattered splats, and three floors
    "wall": lambda rng, n: np.where(rng.random(n) < 0.6, 4.0, rng.uniform(2.0, 6.0, n)),
    "floors": lambda rng, n: rng.choice([2.0, 4.0, 5.5], n),
    # most depths within a few hundred representable values, the rest far away
    "cluster": lambda rng, n: np.where(rng.random(n) < 0.9, 4.0 + rng.integers(0, 300, n) * 4.8e-7, rng.uniform(2.0, 9.0, n)),
}
LENGTHS = [1, 64, 65, 2047, 2048, 2049, 4607, 4608, 4609, 9216, 9217, 16384, 16385, 70000]


def test_the_lists_have_the_lengths_they_are_named_after():
    for n in LENGTHS:
        for depths in DEPTHS.values():
            params, cam = heap(n, depths)
            ranges = oracle.forward(params, cam, W, H)["lists"].ranges.astype(np.int64)
            lengths = ranges[:, 1] - ranges[:, 0]
            assert lengths.max() == n == lengths.sum()


@pytest.mark.gpu
@pytest.mark.parametrize("depths", sorted(DEPTHS))
@pytest.mark.parametrize("n", LENGTHS)
def test_one_list(n, depths):
    params, cam = heap(n, DEPTHS[depths])
    r = _check(params, cam, W, H, cap=max(n, 64))
    assert r.layout.bin_sort_launches == 4


def bin_ms(n, depths):
    """Median device time of gs_bin_sort for one list of n pairs."""
    from tests.gpu_common import gpu_render, torch_mods
    torch, api = torch_mods()
    params, cam = heap(n, DEPTHS[depths])
    r, g, cams, _ = gpu_render(params, cam, W, H, cap=n)
    times = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        api.gs_project(r.cfg, g, cams, r.ws)
        a.record()
        api.gs_bin_sort(r.cfg, r.ws)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return float(np.median(times))


@pytest.mark.gpu
@pytest.mark.parametrize("depths", ["equal", "wall", "floors"])
def test_equal_depths_cost_little_more(depths):
    # (20000 pairs through a network of compare-exchanges of one block: more than 15 times as long)
    assert bin_ms(20000, depths) < 4.0 * bin_ms(20000, "spread")


@pytest.mark.gpu
def test_many_blocks_share_a_giant_list():
    # (one block alone: more than 12 times as long)
    assert bin_ms(300000, "spread") < 5.0 * bin_ms(15000, "spread")
