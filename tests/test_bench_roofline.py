"""The bytes that bench.py credits a binning launch with are those of the binning form that ran, over the live items."""
import types

import numpy as np
import pytest
import torch

import bench


class _Rasterizer:
    def __init__(self, project_launches, live, total):
        self.layout = types.SimpleNamespace(project_launches=project_launches, sort_passes=2, tiles_x=40, tiles_y=30)
        mask = np.zeros((total + 31) // 32 * 32, np.uint8)
        mask[:live] = 1
        self._mask = torch.as_tensor(np.packbits(mask).view(np.int32).copy())

    def ws_view(self, name, dtype, count):
        assert name == "live_mask" and dtype == torch.int32 and count == self._mask.numel()
        return self._mask


@pytest.mark.parametrize("launches,want", [(1, 700 * 64 + 5000 * 44 + 2 * 1200 * 8), (2, 700 * 88 + 5000 * (12 + 48 + 8))])
def test_binning_bytes(monkeypatch, launches, want):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: types.SimpleNamespace(multi_processor_count=152))
    s = types.SimpleNamespace(N=1000, K=2, W=640, H=480)
    roof = bench.roofline("bin_sort", [1.0], {"evals": 0, "evals_bwd": 0}, 5000, s, _Rasterizer(launches, 700, 2000), "none")
    assert roof["achieved"] * 1e6 == pytest.approx(want)
