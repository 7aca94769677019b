"""Binning of camera sets with thousands of super-tiles.

The emission counts the pairs per super-tile in shared memory up to 12288 super-tiles,
beside its lists (about 10 KB, together more than the 48 KB that a launch gets without
asking), and in global memory beyond. Every list against the oracle replica's, just
below and inside the range where both together pass 48 KB, at its end and beyond, for
masks of one word (free layouts: 4 x 4 tiles a super-tile here) and of two (slots), for
the scenes that one block or cluster counts and for those of the general path.
"""
import math

import numpy as np
import pytest

from paper_2505_24053_gb300 import workloads as wl
from tests.test_gpu_forward import _expand_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    return geer


def _scene(n):
    rng = np.random.default_rng(n)
    v = rng.normal(0, 1, (n, 3))
    v *= rng.uniform(2, 5, (n, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
    return wl.Scene(v.astype(np.float32), np.exp(rng.normal(-2.0, 0.5, (n, 3))).astype(np.float32),
                    rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.2, 0.9, n).astype(np.float32),
                    rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)


def _columns(n, supers):
    """n cameras of one column of tiles, `supers` super-tiles high, all around."""
    cams = []
    for i in range(n):
        R, t = wl.pose(wl.rot_y(2 * math.pi * i / n), (0.02 * math.sin(i), 0.0, 0.0))
        cams.append(wl.Camera(wl.EQUIDISTANT, 16, 64 * supers, 2 * math.pi / 3 / (4 * supers), R_cw=R, t_cw=t))
    return cams


def _check(ws, orc, scene, cams, tile_of):
    P, _ = ws.pair_counts()
    k, v = ws.debug_pairs(cap=P)
    ek, ev = _expand_pairs(orc, scene, cams)
    tile = tile_of[(ek >> np.uint64(32)).astype(np.int64)]
    ek = (tile.astype(np.uint64) << np.uint64(32)) | (ek & np.uint64(0xffffffff))
    assert P == ek.size > 0
    assert np.array_equal(k, ek) and np.array_equal(v, ev)


@pytest.mark.parametrize("n", [60, 200], ids=["small_front", "general"])
@pytest.mark.parametrize("ncams,supers", [(245, 40), (246, 40), (250, 40), (256, 48), (256, 49)],
                         ids=["9800", "9840", "10000", "12288", "12544"])
def test_free_layout(geer, orc, n, ncams, supers):
    scene, cams = _scene(n), _columns(ncams, supers)
    assert (ncams * n <= 32768) == (n == 60)
    r = geer.Renderer(cams, n, 0, pair_capacity=1 << 21)
    r.prepare(geer.Gaussians.from_scene(scene))
    _check(r.ws, orc, scene, cams, np.arange(ncams * 4 * supers))


@pytest.mark.parametrize("n", [500, 5000], ids=["small_front", "general"])
@pytest.mark.parametrize("slots,slot_tiles", [(8, 9600), (9, 9600), (10, 9600), (64, 1528), (64, 1536)],
                         ids=["9608", "10809", "12010", "12288", "12352"])
def test_slots(geer, orc, n, slots, slot_tiles):
    scene = _scene(n)
    n_active = 2 if slots == 64 else slots
    cams = []
    for i in range(slots):
        R, t = wl.pose(wl.rot_y(0.7 * i), (0.0, 0.05 * i, 0.0))
        cams.append(wl.Camera(wl.EQUIDISTANT, 150 + 7 * i % 90, 100 + 11 * i % 60, math.radians(150), R_cw=R, t_cw=t))
    active = [i % (slots // n_active) == 0 for i in range(slots)]
    cap = wl.Camera(wl.PINHOLE, 16 * slot_tiles, 16, math.radians(60))
    ws = geer.Workspace([cap] * slots, n, 0, 1 << 21)
    ws.set_camera_slots(cams, active, slot_tiles, slot_tiles * 256)
    ws.preprocess(geer.Gaussians.from_scene(scene))
    ws.bin_sort()
    tile_of, items = [], []
    for i, c in enumerate(cams):
        if active[i]:
            tiles = ((c.width + 15) // 16) * ((c.height + 15) // 16)
            tile_of.append(i * slot_tiles + np.arange(tiles))
            items.append(i)
    P, _ = ws.pair_counts()
    k, v = ws.debug_pairs(cap=P)
    ek, ev = _expand_pairs(orc, scene, [cams[i] for i in items])
    tile = np.concatenate(tile_of)[(ek >> np.uint64(32)).astype(np.int64)]
    ek = (tile.astype(np.uint64) << np.uint64(32)) | (ek & np.uint64(0xffffffff))
    ev = (np.asarray(items)[ev // n] * n + ev % n).astype(np.uint32)
    assert P == ek.size > 0
    assert np.array_equal(k, ek) and np.array_equal(v, ev)
