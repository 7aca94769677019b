"""The order in which the renders take the tiles of one cost bucket.

With n blocks of 1024 tiles the tiles k, k + n, k + 2 n, ... come together, block k after
block k - 1, so that tiles rendered at the same time lie apart in the image and the sums
of a Gaussian over many tiles meet its parts from all over it (neighbouring tiles in turn
moved the gradients of needles near a camera by several times what equal runs differ by).
The order is not part of the interface: it is found in the workspace as a run of words that
is a permutation of the tiles. tile mod n may fall only from one of the 129
buckets to the next.
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


def _orders(ws, n):
    """Every 256-byte aligned run of n words of the workspace that is a permutation of [0, n)."""
    base = (-ws.buf.data_ptr()) % 256
    w = ws.buf[base:base + (ws.buf.numel() - base) // 256 * 256].view(torch.int32)
    at = torch.arange(0, w.numel() - n, 64, device=w.device)
    mine = (w >= 0) & (w < n)
    for value, total in ((mine.long(), n), (torch.where(mine, w, 0).long(), n * (n - 1) // 2)):
        runs = torch.cat([torch.zeros(1, dtype=torch.long, device=w.device), value.cumsum(0)])
        at = at[runs[at + n] - runs[at] == total]
    runs = [w[a:a + n].cpu().numpy() for a in at.tolist()]
    return [v for v in runs if np.array_equal(np.sort(v), np.arange(n))]


@pytest.mark.parametrize("sizes", [[(1440, 1430)], [(640, 500), (777, 333), (1000, 640)], [(512, 512)]],
                         ids=["one", "three", "one_block"])
def test_tiles_of_a_bucket(geer, sizes):
    n = 3000
    rng = np.random.default_rng(2)
    scene = wl.Scene(rng.uniform(-2, 2, (n, 3)).astype(np.float32), np.exp(rng.normal(-3, 0.7, (n, 3))).astype(np.float32),
                     rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.1, 0.9, n).astype(np.float32),
                     rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    cams = []
    for i, (w, h) in enumerate(sizes):
        R, t = wl.pose(wl.rot_y(1.1 * i), (0.0, 0.0, 0.1 * i))
        cams.append(wl.Camera(wl.EQUIDISTANT, w, h, math.radians(170), R_cw=R, t_cw=t))
    tiles = sum(((w + 15) // 16) * ((h + 15) // 16) for w, h in sizes)
    blocks = (tiles + 1023) // 1024
    assert blocks == {1: 8, 3: 5}.get(len(sizes), 0) or tiles == 1024
    torch.cuda.empty_cache()  # (a workspace of an earlier test may leave its order in memory that is not written)
    r = geer.Renderer(cams, n, 0)
    g = geer.Gaussians.from_scene(scene)
    r.forward(g)
    orders = _orders(r.ws, tiles)
    assert orders
    for order in orders:
        k = order % blocks
        assert int((k[1:] < k[:-1]).sum()) <= 128
