"""The per-Gaussian kernels and the binning at the edges of their blocks.

- Rows of SH coefficients copied and written back 16 bytes a lane by whole warps:
  ragged last warps, every degree, gradients written and added (rows of Gaussians
  without a gradient untouched), against the oracle with the tolerance of
  test_gpu_backward.py.
- More cameras than the 32 whose visibility a Gaussian's thread keeps in a word.
- Lists of Gaussians whose association is several rectangles (boxes of more than 32
  super-tiles, several cameras) and item counts around a block, against the replica.
- More block counts than one step of the scan takes (4096).
- Tiles of few entries, walked without bounds, against the same tile with entries that
  no ray hits behind them.
- The binning of small scenes by one block or a cluster against the general path, over
  the items a thread holds, cameras, equal depths and culled Gaussians.
"""
import math

import numpy as np
import pytest
import torch

from paper_2505_24053_gb300 import workloads as wl
from tests.test_gpu_backward import BLOCKS, _compare, _oracle_grads, _scene
from tests.test_gpu_forward import _expand_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    return geer


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 63, 65, 97])
@pytest.mark.parametrize("ncams", [1, 2])
def test_ragged_rows(geer, orc, n, deg, ncams):
    scene = _scene(100 * deg + n, n, deg)
    scene.mean[1::3, 2] *= -1.0  # behind the camera: no gradient
    cams = [wl.Camera(wl.PINHOLE, 40, 32, math.radians(70)), wl.Camera(wl.PINHOLE, 24, 24, math.radians(60))][:ncams]
    dL = np.random.default_rng(n).normal(0, 1, (sum(c.pixels for c in cams), 3)).astype(np.float32)
    r = geer.Renderer(cams, n, deg)
    g = geer.Gaussians.from_scene(scene)
    r.forward(g)
    dL_gpu = torch.as_tensor(dL, device="cuda")
    new = r.backward(g, dL_gpu)
    _compare({k: new[k].cpu().numpy().astype(np.float64) for k in BLOCKS}, _oracle_grads(orc, scene, cams, dL), "new")
    # added to 1: one FP32 addition of the same gradient, itself reproducible to 1e-3 of its largest value
    r.forward(g)
    ones = r.backward(g, dL_gpu, {k: torch.ones_like(v) for k, v in new.items()})
    dead = torch.as_tensor(r.ws.debug_preprocess()[3].reshape(ncams, n).sum(0) == 0, device="cuda")
    for k in BLOCKS:
        big = float(new[k].abs().max())
        assert float((ones[k] - 1 - new[k]).abs().max()) <= 1e-3 * big + 2.0 ** -23 * (1 + big), k
        assert bool((ones[k][dead] == 1).all()) and bool((new[k][dead] == 0).all()), k


def test_more_cameras_than_a_word(geer, orc):
    n = 40
    scene = _scene(3, n, 1)
    cams = []
    for i in range(35):
        R, t = wl.pose(wl.rot_y(2 * math.pi * i / 35), (0.1, 0.0, -0.1))
        cams.append(wl.Camera(wl.PINHOLE, 16, 16, math.radians(60), R_cw=R, t_cw=t))
    dL = np.random.default_rng(1).normal(0, 1, (sum(c.pixels for c in cams), 3)).astype(np.float32)
    r = geer.Renderer(cams, n, 1)
    g = geer.Gaussians.from_scene(scene)
    r.forward(g)
    seen = r.ws.debug_preprocess()[3].reshape(35, n) > 0
    assert seen[:32].any() and seen[32:].any()
    new = r.backward(g, torch.as_tensor(dL, device="cuda"))
    _compare({k: new[k].cpu().numpy().astype(np.float64) for k in BLOCKS}, _oracle_grads(orc, scene, cams, dL), "35")


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 513])
@pytest.mark.parametrize("px,ncams", [(640, 1), (320, 2)])
def test_lists_of_several_rectangles(geer, orc, n, px, ncams):
    rng = np.random.default_rng(n)
    mean = rng.normal(0, 1, (n, 3))
    mean[:, 2] *= 0.2  # near the plane where both angles pass 90 degrees
    mean *= (1.5 + rng.uniform(0, 2, (n, 1))) / np.linalg.norm(mean, axis=1, keepdims=True)
    scene = wl.Scene(mean.astype(np.float32), np.exp(rng.normal(-2.0, 0.6, (n, 3))).astype(np.float32),
                     rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.1, 0.9, n).astype(np.float32),
                     rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    R, t = wl.pose(wl.rot_y(1.0), (0.0, 0.1, 0.0))
    cams = [wl.Camera(wl.EQUIDISTANT, px, px - 13, math.radians(210)),
            wl.Camera(wl.EQUIDISTANT, px - 40, px, math.radians(195), R_cw=R, t_cw=t)][:ncams]
    r = geer.Renderer(cams, n, 0, pair_capacity=1 << 22)
    r.prepare(geer.Gaussians.from_scene(scene))
    P, _ = r.ws.pair_counts()
    k, v = r.ws.debug_pairs(cap=P)
    ek, ev = _expand_pairs(orc, scene, cams)
    assert P == ek.size and np.array_equal(k, ek) and np.array_equal(v, ev)


@pytest.mark.parametrize("w,h", [(132, 3), (3, 132), (140, 131), (64, 64), (71, 70), (120, 110)],
                         ids=["33x1", "1x33", "35x33", "16x16", "15x14", "15x14wide"])
@pytest.mark.parametrize("culled", [0, 33_000], ids=["small_front", "general"])
def test_several_rectangles_over_many_super_tiles(geer, orc, w, h, culled):
    """Items of several rectangles over more than 32 super-tile columns, rows or both (4 x 4 tiles
    each), and over super-tiles of 5 x 5 and 8 x 8 tiles, the latter with masks of two words."""
    n = 40
    rng = np.random.default_rng(w + h)
    v = rng.normal(0, 1, (n, 3))
    v *= rng.uniform(0.3, 6, (n, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
    pad = lambda a: np.concatenate([a, np.repeat(a[:1], culled, 0)]).astype(np.float32)  # noqa: E731
    scene = wl.Scene(pad(v), pad(np.exp(rng.normal(-1.5, 1.0, (n, 3)))), pad(rng.standard_normal((n, 4))),
                     pad(rng.uniform(0.2, 0.9, n)), pad(rng.normal(0, 0.3, (n, 1, 3))), 0)
    scene.scale[n:] = 0.0
    cams = [wl.Camera(wl.EQUIDISTANT, 16 * w - 5, 16 * h - 7, math.radians(230), math.radians(215))]
    r = geer.Renderer(cams, n + culled, 0, pair_capacity=1 << 21)
    r.prepare(geer.Gaussians.from_scene(scene))
    P, _ = r.ws.pair_counts()
    k, val = r.ws.debug_pairs(cap=P)
    first = wl.Scene(scene.mean[:n], scene.scale[:n], scene.quat[:n], scene.opacity[:n], scene.sh[:n], 0)
    ek, ev = _expand_pairs(orc, first, cams)
    assert P == ek.size > 0
    assert np.array_equal(k, ek) and np.array_equal(val, ev)


def test_more_block_counts_than_a_scan_step(geer):
    """4097 blocks of Gaussians: every live item in its tiles' lists, in depth order."""
    n = 4096 * 256 + 17
    rng = np.random.default_rng(8)
    mean = np.stack([rng.uniform(-2, 2, n), rng.uniform(-2, 2, n), rng.uniform(1, 6, n)], 1)
    scene = wl.Scene(mean.astype(np.float32), np.full((n, 3), 1e-3, np.float32),
                     np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.full(n, 0.5, np.float32),
                     np.zeros((n, 1, 3), np.float32), 0)
    cams = [wl.Camera(wl.PINHOLE, 64, 64, math.radians(90)), wl.Camera(wl.PINHOLE, 48, 64, math.radians(80))]
    r = geer.Renderer(cams, n, 0, pair_capacity=1 << 22)
    r.prepare(geer.Gaussians.from_scene(scene))
    counts = r.ws.debug_preprocess()[3]
    P, _ = r.ws.pair_counts()
    k, v = r.ws.debug_pairs(cap=P)
    assert P == k.size == counts.sum(dtype=np.int64)
    assert np.array_equal(np.bincount(v, minlength=2 * n), counts)
    assert (k[1:] >= k[:-1]).all()


def test_more_sort_tiles_than_blocks(geer):
    """More live items and (super-tile, item) pairs than the 3.7M keys that one
    round of the histogram's blocks takes on 152 SMs. Depth order inside each tile,
    equal depths (the same camera twice) in item order."""
    n = 1_100_000
    rng = np.random.default_rng(9)
    z = rng.uniform(1, 6, n)
    mean = np.stack([rng.uniform(-0.4, 0.4, n) * z, rng.uniform(-0.4, 0.4, n) * z, z], 1)
    scene = wl.Scene(mean.astype(np.float32), np.full((n, 3), 1e-3, np.float32),
                     np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.full(n, 0.5, np.float32),
                     np.zeros((n, 1, 3), np.float32), 0)
    r = geer.Renderer([wl.Camera(wl.PINHOLE, 128, 128, math.radians(60))] * 4, n, 0, pair_capacity=1 << 23)
    r.prepare(geer.Gaussians.from_scene(scene))
    counts = r.ws.debug_preprocess()[3]
    P, supers = r.ws.pair_counts()
    assert supers > 3_800_000
    k, v = r.ws.debug_pairs(cap=P)
    assert P == k.size == counts.sum(dtype=np.int64)
    assert np.array_equal(np.bincount(v, minlength=4 * n), counts)
    assert (k[1:] >= k[:-1]).all()
    same = k[1:] == k[:-1]
    assert same.any() and (v[1:][same] > v[:-1][same]).all()


@pytest.mark.parametrize("n,ncams", [(1, 1), (31, 1), (1024, 1), (1025, 1), (341, 3), (4096, 1), (2049, 2), (4097, 1),
                                     (2731, 3), (8192, 1), (16384, 1), (16385, 1),
                                     (32768, 1)])
@pytest.mark.parametrize("fov", [80, 205])
def test_small_front_equals_the_general_path(geer, n, ncams, fov):
    """At most 32768 items are binned by one block or a cluster; the same scene with culled
    Gaussians behind it takes the general path. Same lists, in the same order."""
    rng = np.random.default_rng(n + fov)
    mean = rng.uniform(-2, 2, (n, 3)).astype(np.float32)
    mean[n // 2:] = mean[:n - n // 2]  # equal depths
    opacity = rng.uniform(0.1, 0.9, n).astype(np.float32)
    opacity[::7] = 0.001  # culled
    opacity[0] = 0.9
    scene = wl.Scene(mean, np.exp(rng.normal(-4.0, 0.8, (n, 3))).astype(np.float32),
                     rng.standard_normal((n, 4)).astype(np.float32), opacity,
                     rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    pad = 32769
    big = wl.Scene(*(np.concatenate([a, np.resize(a, (pad,) + a.shape[1:])]) for a in
                     (scene.mean, scene.scale, scene.quat)),
                   np.concatenate([opacity, np.zeros(pad, np.float32)]),
                   np.concatenate([scene.sh, np.zeros((pad, 1, 3), np.float32)]), 0)
    cams = []
    for i in range(ncams):
        R, t = wl.pose(wl.rot_y(1.3 * i), (0.1 * i, 0.0, 0.0))
        cams.append(wl.Camera(wl.EQUIDISTANT, 150 + 20 * i, 130, math.radians(fov), R_cw=R, t_cw=t))
    lists = []
    for sc in (scene, big):
        r = geer.Renderer(cams, sc.n, 0, pair_capacity=1 << 21)
        rgb = r.forward(geer.Gaussians.from_scene(sc))
        P, supers = r.ws.pair_counts()
        k, v = r.ws.debug_pairs(cap=P)
        lists.append((P, supers, r.ws.live_items(), k, v // sc.n, v % sc.n, rgb.cpu().numpy()))
    assert lists[0][:3] == lists[1][:3]
    for a, b in zip(lists[0][3:], lists[1][3:]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 12])
@pytest.mark.parametrize("splat", [False, True])
def test_tiles_of_few_entries(geer, n, splat):
    rng = np.random.default_rng(n)
    fov = math.radians(60)
    cam = wl.Camera(wl.PINHOLE, 16, 16, fov)
    i = rng.integers(1, 16, (40, 2))
    ang = (i / 16 - 0.5) * fov  # between the rays, which lie at ((i + 1/2) / 16 - 1/2) fov
    far = np.stack([np.tan(ang[:, 0]) * 20, np.tan(ang[:, 1]) * 20, np.full(40, 20.0)], 1)
    near = np.stack([rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.uniform(3, 5, n)], 1)
    quat = rng.standard_normal((n + 40, 4)).astype(np.float32)
    scene = wl.Scene(np.concatenate([near, far]).astype(np.float32),
                     np.concatenate([np.exp(rng.normal(-1.5, 0.5, (n, 3))), np.full((40, 3), 1e-4)]).astype(np.float32),
                     quat, np.concatenate([rng.uniform(0.2, 0.9, n), np.full(40, 0.9)]).astype(np.float32),
                     rng.normal(0, 0.3, (n + 40, 1, 3)).astype(np.float32), 0)
    prm = geer.params_c(alpha_model=geer.ALPHA_SPLAT) if splat else None
    images = []
    for sc in (scene.subset(np.arange(n)), scene):
        r = geer.Renderer([cam], sc.n, 0, params=prm)
        T = torch.empty(256, device="cuda")
        images.append((r.forward(geer.Gaussians.from_scene(sc), T=T), T, r.ws.pair_counts()[0]))
    assert images[0][2] <= n and images[1][2] >= images[0][2] + 30
    assert torch.equal(images[0][0], images[1][0]) and torch.equal(images[0][1], images[1][1])
    assert float(images[0][1].min()) < 0.9
