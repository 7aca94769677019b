"""The optimiser step, the refinement's copies and the image metrics at the edges of
their blocks.

The first two are elementwise: an Adam step of n Gaussians gives bit for bit what the same
Gaussians get inside a larger array (the groups start at every alignment of the flat
moments), and the refinement moves rows unchanged. The metrics are compared with the
oracle within test_gpu_eval.py's tolerance.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geer():
    from paper_2505_24053_gb300 import geer
    geer.lib()
    return geer


NAMES = ("mean", "log_scale", "quat", "logit_opacity", "sh")


def _raw(rng, n, deg):
    k = (deg + 1) ** 2
    raw = {"mean": rng.normal(0, 1, (n, 3)), "log_scale": rng.normal(-2, 0.5, (n, 3)), "quat": rng.normal(0, 1, (n, 4)),
           "logit_opacity": rng.normal(0, 1.5, n), "sh": rng.normal(0, 0.3, (n, k, 3))}
    return {key: v.astype(np.float32) for key, v in raw.items()}


def _groups(flat, n, k):
    return [p.reshape(n, -1) for p in np.split(flat, np.cumsum([3 * n, 3 * n, 4 * n, n]))]


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 85, 341, 342, 1023, 1024, 1025])
def test_adam_of_part_of_an_array(geer, n, deg):
    big, k = 1600, (deg + 1) ** 2
    rng = np.random.default_rng(10 * n + deg)
    raw = _raw(rng, big, deg)
    grad = dict(zip(("mean", "scale", "quat", "opacity", "sh"), _raw(rng, big, deg).values()))
    out = []
    for c in (n, big):
        a = geer.Adam(*(raw[key][:c] for key in NAMES), deg, lr_mean=1e-3)
        for _ in range(2):
            a.step({key: torch.as_tensor(np.ascontiguousarray(v[:c]), device="cuda") for key, v in grad.items()})
        out.append([a.raw[key].cpu().numpy().reshape(c, -1)[:n] for key in NAMES] +
                   [p[:n] for q in (a.m, a.v) for p in _groups(q.cpu().numpy(), c, k)] +
                   [a.gaussians.scale.cpu().numpy()[:n], a.gaussians.opacity.cpu().numpy()[:n]])
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 700])
def test_refinement_moves_rows(geer, n, deg):
    k = (deg + 1) ** 2
    rng = np.random.default_rng(n + deg)
    raw = _raw(rng, n, deg)
    act = rng.integers(0, 4, n)  # prune, keep, clone, split
    act[0] = 2
    raw["logit_opacity"] = np.where(act == 0, np.float32(-9), np.clip(raw["logit_opacity"], -2, 2)).astype(np.float32)
    raw["log_scale"] = np.where(act[:, None] == 3, np.float32(0), np.float32(-6)) + 0.1 * np.tanh(raw["log_scale"])
    raw["log_scale"] = raw["log_scale"].astype(np.float32)
    a = geer.Adam(*(raw[key] for key in NAMES), deg)
    a.m.copy_(torch.as_tensor(rng.normal(0, 1, a.m.shape), device="cuda"))
    a.v.copy_(torch.as_tensor(rng.uniform(0, 1, a.v.shape), device="cuda"))
    m0, v0 = (_groups(q.cpu().numpy().copy(), n, k) for q in (a.m, a.v))
    accum = torch.as_tensor(np.where(act >= 2, 1.0, 0.0), dtype=torch.float32, device="cuda")
    z = torch.as_tensor(rng.normal(0, 1, (n, 2, 3)), dtype=torch.float32, device="cuda")
    a.densify(accum, torch.ones_like(accum), z, clone_max_scale=0.1)
    src = np.repeat(np.arange(n), np.array([0, 1, 2, 2])[act])
    second = np.concatenate([[False], src[1:] == src[:-1]])
    split = act[src] == 3
    for key in NAMES:
        got, want = a.raw[key].cpu().numpy().reshape(src.size, -1), raw[key].reshape(n, -1)[src]
        same = ~split if key in ("mean", "log_scale") else np.ones_like(split)
        assert np.array_equal(got[same], want[same]), key
    for q, q0 in ((a.m, m0), (a.v, v0)):
        for got, want in zip(_groups(q.cpu().numpy(), src.size, k), q0):
            assert np.array_equal(got, np.where((second | split)[:, None], np.float32(0), want[src]))


@pytest.mark.parametrize("w", [1, 31, 32, 33, 65])
@pytest.mark.parametrize("h", [1, 15, 16, 17, 34])
def test_metrics_at_tile_edges(geer, h, w):
    from oracle import metrics as M
    rng = np.random.default_rng(100 * h + w)
    pred, gt = (rng.uniform(0, 1, (h, w, 3)).astype(np.float32) for _ in range(2))
    regions = rng.integers(0, 4, (h, w)).astype(np.uint8)
    regions[regions == 3] = 255
    res = geer.image_metrics(*(torch.as_tensor(x, device="cuda") for x in (pred, gt, regions)), 3)
    ref = M.region_metrics(pred, gt, regions, 3)
    for r in range(3):
        assert res[r]["count"] == int(ref[r, 2])
        assert abs(res[r]["sse"] - ref[r, 0]) <= 1e-5 * ref[r, 0] + 1e-9
        assert abs(res[r]["ssim_sum"] - ref[r, 1]) <= 1e-5 * ref[r, 2]
