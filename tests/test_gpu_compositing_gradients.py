"""Gradients of the compositing's two per-splat forms against the oracle, for every splat set of
test_gpu_compositing_paths: no upstream gradient where a decision lies within rounding of its threshold."""
import numpy as np
import pytest

import oracle
from scenes import random_image

from tests.gpu_common import GRAD_RTOL, check_images, gpu_render, rel_l2, to_np, torch_mods
from tests.test_gpu_compositing_paths import _splats

CASES = [(logit, offset, thin) for logit in (-2.0, 3.5, 4.2, 8.0) for offset in (0.0, 1e-3, 0.25) for thin in (False, True)]


def _case(logit, offset, thin):
    params, cam, W, H = _splats(logit, offset, thin)
    orc = oracle.forward(params, cam, W, H)
    clear = orc["near"] == 0
    gr, gd = random_image(41, (1, 3, H, W)) * clear[:, None], random_image(42, (1, H, W)) * clear
    return params, cam, W, H, orc, clear, gr.astype(np.float32), gd.astype(np.float32)


def test_most_pixels_take_part():
    for case in CASES:
        _, _, _, _, orc, clear, _, _ = _case(*case)
        assert clear.mean() > 0.9 and (orc["near"] >= 2).mean() < 1e-2, case


@pytest.mark.gpu
@pytest.mark.parametrize("logit,offset,thin", CASES)
def test_gradients(logit, offset, thin):
    torch, _ = torch_mods()
    params, cam, W, H, orc, _, gr, gd = _case(logit, offset, thin)
    og = oracle.backward(params, cam, W, H, orc["lists"], gr, gd)
    r, g, ct, out = gpu_render(params, cam, W, H, cap=1 << 16)
    check_images(to_np(out), orc, max_excluded=1e-2)
    for px in (0, 1, 2, 4):
        r.cfg.fwd_px_per_thread = r.cfg.bwd_px_per_thread = px
        out = r.render(g, ct)
        grads = to_np(r.backward(g, ct, out, torch.as_tensor(gr).cuda(), torch.as_tensor(gd).cuda()))
        for k in ("means", "log_scales", "quats", "opacity_logits", "rgb", "pose"):
            assert rel_l2(grads[k], og[k]) < GRAD_RTOL, (px, k)
