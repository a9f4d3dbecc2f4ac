"""The compositing's two per-splat forms (with and without the clamp and power tests) on splats made to need
them: opacities above and below the clamp, means exactly on and just beside pixel centres, round and needle-thin
splats; images and gradients against the oracle, and every pixels-per-thread value alike."""
import numpy as np
import pytest

import oracle
from scenes import random_image
from scenes.generate import camera_array

from gpu_common import GRAD_RTOL, check_images, gpu_render, rel_l2, to_np, torch_mods

pytestmark = pytest.mark.gpu


def _splats(logit, offset, thin, n=60, W=80, H=48, f=32.0):
    rng = np.random.default_rng(7)
    z = rng.integers(8, 24, n) / 4.0  # exact in binary, so means land exactly on pixel centres
    uv = np.stack([rng.integers(0, W, n), rng.integers(0, H, n)], 1) + 0.5 + offset
    means = np.concatenate([(uv - [W / 2, H / 2]) * z[:, None] / f, z[:, None]], 1).astype(np.float32)
    scales = rng.uniform(-1.5, 0.3, (n, 3))
    if thin:
        scales[:, 1:] = -6.0
    quats = rng.normal(size=(n, 4))
    params = (means, scales.astype(np.float32), quats.astype(np.float32), np.full(n, logit, np.float32),
              rng.uniform(0, 1, (n, 3)).astype(np.float32))
    return params, camera_array(f, f, W / 2, H / 2, np.eye(3), np.zeros(3)), W, H


@pytest.mark.parametrize("thin", [False, True])
@pytest.mark.parametrize("offset", [0.0, 1e-3, 0.25])
@pytest.mark.parametrize("logit", [-2.0, 3.5, 4.2, 8.0])
def test_checked_and_plain_splats(logit, offset, thin):
    torch, api = torch_mods()
    params, cam, W, H = _splats(logit, offset, thin)
    orc = oracle.forward(params, cam, W, H)
    r, g, ct, out = gpu_render(params, cam, W, H, cap=1 << 16)
    first = to_np(out)
    # (a mean exactly on a pixel centre has power 0 there: its sign is within the guard band)
    check_images(first, orc, max_excluded=1.0 if offset == 0.0 else 1e-2)
    gr, gd = random_image(41, (1, 3, H, W)), random_image(42, (1, H, W))
    og = oracle.backward(params, cam, W, H, orc["lists"], gr, gd)
    for px in (0, 1, 2, 4):
        r.cfg.fwd_px_per_thread = r.cfg.bwd_px_per_thread = px
        out = r.render(g, ct)
        for k, v in to_np(out).items():
            assert np.array_equal(v, first[k]), (px, k)
        grads = to_np(r.backward(g, ct, out, torch.as_tensor(gr).cuda(), torch.as_tensor(gd).cuda()))
        if offset == 0.25 and (orc["near"] == 0).all():  # no decision within rounding of its threshold
            for k in ("means", "log_scales", "quats", "opacity_logits", "rgb", "pose"):
                assert rel_l2(grads[k], og[k]) < GRAD_RTOL, (px, k)
