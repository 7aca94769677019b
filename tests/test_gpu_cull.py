"""The forward's list filters and sub-tile bounds.

- The bound that lets a warp skip a list entry never drops one that a ray of it
  hits: the checked build walks the dropped entries too and records a violation
  (site 8) when a ray hits one. Scenes: specks below the ray spacing (tested at
  every ray), needles and flakes (thin conics, non-convex quadratics), blobs
  around the camera (conics across 90 degrees), on cameras from 60 to 210 degrees,
  ragged images, the exact integral and the splat alpha. The checked build's image
  is libgeer.so's bit for bit.
- Every tile's list equals the oracle replica's association for every super-tile
  size (tile masks of one and of two words, one and two sort passes), with and
  without rays beyond 90 degrees.
- A sparse tile of a long super-tile list (the scan that skips empty groups):
  its list against the replica, and its pixels bit for bit those of a scene that
  holds only its own Gaussians.
"""
import math

import numpy as np
import pytest
import torch

from paper_2505_24053_gb300 import workloads as wl
from tests.test_gpu_forward import _expand_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    geer.lib(checked=True)
    return geer


def _scene(kind, n, seed):
    rng = np.random.default_rng(seed)
    mean = rng.uniform(-3, 3, (n, 3))
    log_s = {"specks": rng.normal(-6.5, 0.6, (n, 3)),
             "needles": np.stack([rng.normal(-1.5, 0.5, n), rng.normal(-6, 0.5, n), rng.normal(-6, 0.5, n)], 1),
             "flakes": np.stack([rng.normal(-1.5, 0.5, n), rng.normal(-1.5, 0.5, n), rng.normal(-6, 0.5, n)], 1),
             "blobs": rng.normal(-0.5, 0.4, (n, 3)),
             "mixed": rng.normal(-3.5, 1.5, (n, 3))}[kind]
    return wl.Scene(mean.astype(np.float32), np.exp(log_s).astype(np.float32),
                    rng.standard_normal((n, 4)).astype(np.float32),
                    (1 / (1 + np.exp(-rng.normal(-0.5, 1.5, n)))).astype(np.float32),
                    rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)


CAMS = [wl.Camera(wl.PINHOLE, 150, 110, math.radians(60)), wl.Camera(wl.PINHOLE, 97, 64, math.radians(140)),
        wl.Camera(wl.EQUIDISTANT, 203, 160, math.radians(180)), wl.Camera(wl.EQUIDISTANT, 130, 125, math.radians(210)),
        wl.Camera(wl.KANNALA_BRANDT, 320, 211, math.radians(190), k=wl.kb_coeffs(3))]


@pytest.mark.parametrize("splat", [False, True], ids=["exact", "splat"])
@pytest.mark.parametrize("kind,n", [("specks", 30000), ("needles", 3000), ("flakes", 3000), ("blobs", 400),
                                    ("mixed", 8000)])
def test_no_hit_is_dropped(geer, kind, n, splat):
    scene = _scene(kind, n, 5 + n)
    g = geer.Gaussians.from_scene(scene)
    params = geer.params_c(alpha_model=geer.ALPHA_SPLAT) if splat else None
    for cam in CAMS:
        imgs = []
        for checked in (False, True):
            ws = geer.Workspace([cam], n, 0, 1 << 20, params, library=geer.lib(checked=checked))
            rgb = torch.empty((cam.pixels, 3), device="cuda")
            ws.preprocess(g)
            ws.bin_sort()
            ws.render_fwd(rgb)
            assert ws.bounds_violation() == (0, 0), (kind, cam)
            imgs.append(rgb)
        assert torch.equal(imgs[0], imgs[1]), (kind, cam)


# edges in tiles -> super-tile size: 64 -> 4, 65 -> 5, 81 -> 6, 97 -> 7, 113 -> 8, 129 -> 4 in two passes
@pytest.mark.parametrize("edge,size", [(64, 4), (65, 5), (81, 6), (97, 7), (113, 8), (129, 4)])
@pytest.mark.parametrize("model,fov", [(wl.PINHOLE, 70), (wl.EQUIDISTANT, 200)])
def test_tile_lists_of_every_super_tile_size(geer, orc, edge, size, model, fov):
    cam = wl.Camera(model, 16 * edge - 5, 16 * edge - 9, math.radians(fov))
    tiles = [edge, edge]
    ids = lambda s: math.ceil(tiles[0] / s) * math.ceil(tiles[1] / s)  # noqa: E731
    assert size == next((s for s in range(4, 9) if ids(s) <= 256), 4)
    scene = _scene("mixed", 150, edge)
    scene.scale[:] = np.minimum(scene.scale, 0.1)
    r = geer.Renderer([cam], scene.n, 0, pair_capacity=1 << 21)
    P = r.prepare(geer.Gaussians.from_scene(scene))
    P, _ = r.ws.pair_counts()
    k, v = r.ws.debug_pairs(cap=P)
    ek, ev = _expand_pairs(orc, scene, [cam])
    assert P == ek.size and np.array_equal(k, ek) and np.array_equal(v, ev)


@pytest.mark.parametrize("own", [3, 70, 400])
def test_sparse_tile_of_a_long_list(geer, orc, own):
    """Super-tile (0, 0) of a 128 x 128 pinhole: 120000 specks on its first tile,
    `own` on tile (3, 3), one super-tile list."""
    n = 120_000
    cam = wl.Camera(wl.PINHOLE, 128, 128, math.radians(60))
    rng = np.random.default_rng(own)
    at = (np.arange(n) >= n - own).astype(np.float64)  # the last ones on tile (3, 3)
    px = rng.uniform(3, 12, (n, 2)) + 48.0 * at[:, None]
    ang = ((px + 0.5) / 128 - 0.5) * math.radians(60)
    z = rng.uniform(3, 7, n)
    mean = np.stack([np.tan(ang[:, 0]) * z, np.tan(ang[:, 1]) * z, z], 1)
    scene = wl.Scene(mean.astype(np.float32), np.full((n, 3), 0.004, np.float32),
                     rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.1, 0.9, n).astype(np.float32),
                     rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    perm = rng.permutation(n)
    scene = scene.subset(perm)
    r = geer.Renderer([cam], n, 0)
    rgb = r.forward(geer.Gaussians.from_scene(scene)).view(128, 128, 3)
    P, _ = r.ws.pair_counts()
    k, v = r.ws.debug_pairs(cap=P)
    ek, ev = _expand_pairs(orc, scene, [cam])
    assert P == ek.size and np.array_equal(k, ek) and np.array_equal(v, ev)
    tile = (k >> np.uint64(32)) == 3 * 8 + 3
    assert tile.sum() >= own
    alone = scene.subset(np.sort(v[tile]))
    ra = geer.Renderer([cam], alone.n, 0)
    rgb_a = ra.forward(geer.Gaussians.from_scene(alone)).view(128, 128, 3)
    assert torch.equal(rgb[48:64, 48:64], rgb_a[48:64, 48:64])
