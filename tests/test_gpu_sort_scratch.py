"""gs_sort_pairs in a scratch buffer sized for more pairs than it sorts, across the sizes where the tiles change."""
import pytest

from tests.gpu_common import torch_mods

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sized_for", [(1_000_000, 1_000_001), (700_001, 1_000_000), (900_000, 1_000_001),
                                         (1_000_000, 1_000_000)])
def test_scratch_for_more_pairs_is_enough(n, sized_for):
    torch, api = torch_mods()
    gen = torch.Generator("cuda").manual_seed(n)
    keys = torch.randint(0, 1 << 40, (n,), generator=gen, device="cuda")
    keys[::3] = keys[0]  # equal keys: the sort is stable
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    want, order = torch.sort(keys, stable=True)
    tmp = torch.empty(api.gs_sort_pairs_tmp_size(sized_for), dtype=torch.uint8, device="cuda")
    api.gs_sort_pairs(keys, vals, 40, tmp)
    assert torch.equal(keys, want) and torch.equal(vals.long(), order)
