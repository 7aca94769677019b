"""A dL/dC that is not finite at some pixels.

An infinity or NaN in one channel of a pixel reaches that channel's colour sums (and
sigma's and the geometry's) of the Gaussians that the pixel's ray composites, and
nothing else: the other channels' colour sums, and every sum of the other Gaussians,
are those of the same gradient with zeros there (1e-5 of the column's size, the
reordering of FP32 atomics: test_gpu_fused.py).
"""
import math

import numpy as np
import pytest
import torch

from paper_2505_24053_gb300 import workloads as wl
from tests.test_gpu_backward import _scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    return geer


@pytest.mark.parametrize("splat", [False, True], ids=["exact", "splat"])
@pytest.mark.parametrize("bad", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("channel", [0, 1, 2])
def test_only_its_own_sums(geer, splat, bad, channel):
    n = 600
    scene = _scene(11, n, 1)
    cam = wl.Camera(wl.PINHOLE, 80, 64, math.radians(80))
    prm = geer.params_c(assoc=geer.ASSOC_EWA, snugbox=True, alpha_model=geer.ALPHA_SPLAT) if splat else None
    r = geer.Renderer([cam], n, 1, params=prm)
    g = geer.Gaussians.from_scene(scene)
    pix = [17 * 80 + 40, 18 * 80 + 41, 50 * 80 + 3]

    def sums(dL):
        r.forward(g)
        r.ws.render_bwd_tiles(torch.as_tensor(dL, device="cuda"))
        acc = r.ws.grad_accumulators().clone()
        grads = {k: torch.empty_like(getattr(g, k)) for k in ("mean", "scale", "quat", "opacity", "sh")}
        r.ws.preprocess_bwd(g, grads, accumulate=False)
        return acc, grads

    dL = np.random.default_rng(4).normal(0, 1, (cam.pixels, 3)).astype(np.float32)
    only = np.zeros_like(dL)
    only[pix] = 1.0
    hit = (sums(only)[0][:, 1:4] != 0).any(1)  # the Gaussians that these rays composite
    assert 3 <= int(hit.sum()) <= n - 100
    without, finite = dL.copy(), dL.copy()
    without[pix] = 0.0
    finite[pix, channel] = 0.0  # the other channels of these pixels stay
    dL[pix, channel] = bad
    acc, grads = sums(dL)
    ref, other = sums(without)[0], sums(finite)[0]
    assert not bool(acc[hit][:, 1 + channel].isfinite().any())
    assert bool(acc[~hit].isfinite().all())
    size = ref.abs().amax(0)
    assert bool(((acc - ref)[~hit].abs() <= 1e-5 * size).all())
    for ch in range(3):
        if ch != channel:
            assert bool(((acc - other)[:, 1 + ch].abs() <= 1e-5 * other[:, 1 + ch].abs().max()).all()), ch
            assert bool(grads["sh"][:, :, ch].isfinite().all()), ch


@pytest.mark.parametrize("splat", [False, True], ids=["exact", "splat"])
@pytest.mark.parametrize("coeff,size", [(math.inf, 1.0), (2e37, 1e3)], ids=["inf", "overflow"])
def test_colour_that_overflows(geer, splat, coeff, size):
    """A Gaussian whose colour, or its product with dL/dC, is not finite: the colour sums of every
    Gaussian are weights times dL/dC, so they are those of the same scene with an ordinary colour there."""
    n = 600
    scene = _scene(11, n, 1)
    cam = wl.Camera(wl.PINHOLE, 80, 64, math.radians(80))
    prm = geer.params_c(assoc=geer.ASSOC_EWA, snugbox=True, alpha_model=geer.ALPHA_SPLAT) if splat else None
    r = geer.Renderer([cam], n, 1, params=prm)
    g = geer.Gaussians.from_scene(scene)
    dL = size * torch.randn((cam.pixels, 3), generator=torch.Generator().manual_seed(5)).cuda()

    def sums():
        rgb = r.forward(g).clone()
        r.ws.render_bwd_tiles(dL)
        acc = r.ws.grad_accumulators().clone()
        grads = {k: torch.empty_like(getattr(g, k)) for k in ("mean", "scale", "quat", "opacity", "sh")}
        r.ws.preprocess_bwd(g, grads, accumulate=False)
        return rgb, acc, grads["sh"]

    one = int(sums()[1][:, 1:4].abs().sum(1).argmax())  # a Gaussian that many rays composite
    sh = g.sh.view(n, 4, 3)
    sh[one] = 0.0
    sh[one, 0] = 1.0
    _, ref, ref_sh = sums()
    assert bool(ref.isfinite().all()) and float(ref[one, 1:4].abs().min()) > 0
    sh[one, 0] = coeff
    rgb, acc, dsh = sums()
    assert not bool(acc[:, 0].isfinite().all())  # (sigma's sums and the geometry's do hold the colour)
    assert coeff < math.inf or not bool(rgb.isfinite().all())
    for got, want in ((acc[:, 1:4], ref[:, 1:4]), (dsh.view(n, -1), ref_sh.view(n, -1))):
        assert bool(((got - want).abs() <= 1e-5 * want.abs().amax(0)).all())
