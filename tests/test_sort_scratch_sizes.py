"""gs_sort_pairs accepts scratch that gs_sort_pairs_tmp_size gave for at least as many pairs, at every step of its tile
sizes (the host's decision alone: a stand-in for the CUDA runtime, no GPU)."""
import ctypes

import pytest

from tests.test_launch_errors import faked  # noqa: F401  (fixture)

STEPS = (200_000, 600_000, 1_000_000)


@pytest.mark.parametrize("step", STEPS)
def test_scratch_of_a_larger_sort_is_enough(faked, step):  # noqa: F811
    faked.fake_reset(b"", b"")
    size = ctypes.c_size_t()

    def tmp_size(n):
        assert faked.gs_sort_pairs_tmp_size(ctypes.c_int64(n), ctypes.byref(size)) == 0
        return size.value

    p = ctypes.c_void_p(1 << 20)  # (never read: nothing runs)
    for n in (step // 2, step - 1, step, step + 1, 4 * step // 3):
        for m in (n, n + 1, step + 1, step + 2, 5 * step // 4, 2 * step):
            if m >= n:
                code = faked.gs_sort_pairs(p, p, ctypes.c_int64(n), 40, p, ctypes.c_size_t(tmp_size(m)), None, None)
                assert code == 0, (n, m)
        least = min(tmp_size(m) for m in range(n, 3 * n, max(1, n // 50)))
        assert faked.gs_sort_pairs(p, p, ctypes.c_int64(n), 40, p, ctypes.c_size_t(n * 12), None, None) == 2 and least > n * 12


@pytest.mark.gpu
@pytest.mark.parametrize("n,sized_for", [(200_000, 200_001), (190_000, 200_001), (200_000, 600_001)])
def test_sort_in_that_scratch(n, sized_for):
    from tests.gpu_common import torch_mods
    torch, api = torch_mods()
    gen = torch.Generator("cuda").manual_seed(n)
    keys = torch.randint(0, 1 << 40, (n,), generator=gen, device="cuda")
    keys[::3] = keys[0]  # equal keys: the sort is stable
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    want, order = torch.sort(keys, stable=True)
    api.gs_sort_pairs(keys, vals, 40, torch.empty(api.gs_sort_pairs_tmp_size(sized_for), dtype=torch.uint8, device="cuda"))
    assert torch.equal(keys, want) and torch.equal(vals.long(), order)
