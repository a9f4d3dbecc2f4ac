"""Images wider than 4096 pixels (the tile scan raises its shared-memory limit) and span grids of more than 6144 cells (the
projection counts in global memory): pairs and images equal the oracle's."""
import pytest

import oracle
from scenes import make_scene

from tests.gpu_common import check_images, gpu_render, to_np
from tests.test_gpu_tile_sort import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,K,n", [(4112, 32, 1, 700), (5000, 48, 2, 900), (2000, 1000, 1, 2000), (1600, 1000, 3, 600)])
def test_wide_images_and_large_span_grids(W, H, K, n):
    s = make_scene("window500k", n=n, K=K, W=W, H=H, f=0.8 * min(W, 4 * H))
    _check(s.params(), s.cams, W, H, cap=1 << 18)
    _, _, _, out = gpu_render(s.params(), s.cams, W, H, cap=1 << 18)
    check_images(to_np(out), oracle.forward(s.params(), s.cams, W, H))
