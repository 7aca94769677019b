"""Scales and alphas at the ends of FP32.

- A scene times a power of two is the same image, to 1e-5 (kappa has no length in it;
  every value of the render's chain is scaled by a power of two), from 2^-58 to 2^60,
  where |d_u|^2 nears the ends of the normal numbers (beyond, the squared distances
  leave FP32), and its gradients with respect to mean and scale are divided by it (the
  backward tests' 1e-3).
- Alphas down to alpha_min = 2^-125: |d_u|^2's reciprocal and 2^x keep their relative
  accuracy over the whole range. The exponent argument reaches 125 with a relative error
  of some ten 2^-24 in kappa, so alpha's relative error stays below
  125 ln 2 x 12 x 2^-24 = 6.2e-5: 1e-4. Below alpha_min there is nothing.
"""
import math

import numpy as np
import pytest
import torch

from paper_2505_24053_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    return geer


def _scene(exponent):
    rng = np.random.default_rng(6)
    n, c = 40, 2.0 ** exponent
    mean = np.stack([rng.uniform(-2, 2, n), rng.uniform(-2, 2, n), rng.uniform(6, 12, n)], 1).astype(np.float32)
    scale = np.exp(rng.normal(-1.0, 0.4, (n, 3))).astype(np.float32)
    return wl.Scene((mean * c).astype(np.float32), (scale * c).astype(np.float32),
                    rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.2, 0.9, n).astype(np.float32),
                    rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32), 0)


def _render(geer, exponent):
    cam = wl.Camera(wl.PINHOLE, 70, 50, math.radians(60))
    scene = _scene(exponent)
    r = geer.Renderer([cam], scene.n, 0)
    g = geer.Gaussians.from_scene(scene)
    T = torch.empty(cam.pixels, device="cuda")
    rgb = r.forward(g, T=T)
    dL = torch.as_tensor(np.random.default_rng(1).normal(0, 1, (cam.pixels, 3)).astype(np.float32), device="cuda")
    grads = r.backward(g, dL)
    return rgb, T, {k: grads[k].double() * 2.0 ** (exponent if k in ("mean", "scale") else 0) for k in grads}


@pytest.mark.parametrize("exponent", [-58, -30, 40, 59, 60])
def test_a_scene_times_a_power_of_two(geer, exponent):
    rgb, T, grads = _render(geer, 0)
    rgb2, T2, grads2 = _render(geer, exponent)
    assert float(T.min()) < 0.5
    assert float((rgb2 - rgb).abs().max()) <= 1e-5 and float((T2 - T).abs().max()) <= 1e-5
    for k in grads:
        assert float((grads2[k] - grads[k]).norm()) <= 1e-3 * float(grads[k].norm()), k


def test_faint_alphas(geer):
    s, z, sigma, amin = 0.4, 10.0, 0.5, 2.0 ** -125
    cam = wl.Camera(wl.PINHOLE, 200, 150, math.radians(60))
    scene = wl.Scene(np.float32([[0, 0, z]]), np.full((1, 3), s, np.float32), np.float32([[1, 0, 0, 0]]),
                     np.float32([sigma]), np.full((1, 1, 3), 0.7, np.float32), 0)
    r = geer.Renderer([cam], 1, 0, params=geer.params_c(alpha_min=amin, T_min=0.0))
    cam.bg = (0.0, 0.0, 0.0)
    r.ws.set_cameras([cam])
    rgb = r.forward(geer.Gaussians.from_scene(scene)).cpu().numpy().reshape(150, 200, 3)[..., 0].astype(np.float64)
    fov_y = 2 * math.atan(math.tan(math.radians(30)) * 150 / 200)
    th = ((np.arange(200) + 0.5) / 200 - 0.5) * float(np.float32(math.radians(60)))
    ph = ((np.arange(150) + 0.5) / 150 - 0.5) * fov_y
    d = np.stack(np.broadcast_arrays(np.sin(th)[None] * np.cos(ph)[:, None], np.cos(th)[None] * np.sin(ph)[:, None],
                                     np.cos(th)[None] * np.cos(ph)[:, None]), -1)
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    s32 = float(np.float32(s))
    alpha = sigma * np.exp(-0.5 * (z / s32) ** 2 * (d[..., 0] ** 2 + d[..., 1] ** 2))
    colour = 0.5 + 0.28209479177387814 * float(np.float32(0.7))
    inside, outside = alpha > amin * (1 + 1e-4), alpha < amin * (1 - 1e-4)
    assert alpha[inside].min() < 2.0 ** -120 and outside.any()
    assert np.abs(rgb[inside] / (alpha * colour)[inside] - 1).max() < 1e-4
    assert not rgb[outside].any()
