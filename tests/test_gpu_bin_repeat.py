"""gs_bin_sort called again after one gs_project leaves the same sorted pairs, ranges and images, on both binning forms
and with lists of more than 2048 pairs."""
import pytest

from scenes import make_scene

from tests.gpu_common import gpu_render, torch_mods

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n,K,W,H,f", [("window500k", 3000, 3, 208, 160, 160.0), ("aerial2m", 40000, 1, 208, 192, 20.0),
                                            ("map100k", 2000, 1, 96, 64, 80.0)])
def test_repeated_calls(name, n, K, W, H, f):
    torch, api = torch_mods()
    s = make_scene(name, n=n, K=K, W=W, H=H, f=f)
    r, g, cams, first = gpu_render(s.params(), s.cams, W, H, cap=1 << 18)
    pairs, tiles = r.status()[2], r.K * r.layout.tiles_x * r.layout.tiles_y

    def sorted_pairs():
        return [r.ws_view("keys_sorted", torch.int64, pairs).clone(), r.ws_view("vals_sorted", torch.int32, pairs).clone(),
                r.ws_view("ranges", torch.int32, 2 * tiles).clone()]

    want = sorted_pairs()
    for _ in range(5):
        api.gs_bin_sort(r.cfg, r.ws)
        assert all(torch.equal(a, b) for a, b in zip(sorted_pairs(), want))
    out = r.new_outputs()
    api.gs_raster_fwd(r.cfg, r.ws, out["rgb"], out["depth"], out["T"], out["last"])
    assert all(torch.equal(out[k], first[k]) for k in out) and r.status()[0] == 0
