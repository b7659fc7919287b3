"""Detection where its kernels change course: cell counts around one pass of the offset
scan (16 x 1024 cells), images with candidates at every pixel or nowhere, and orientations
near the bin boundaries (the FP32 angle is used only away from them; every bin must be the
FP64 one)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_03986_gb300 as P
from conftest import to_dev

pytestmark = pytest.mark.gpu


def _detect(ctx, img, w, h, t, max_kps):
    kps, cnt = ctx.detect(to_dev(img), w, h, t, max_kps)
    torch.cuda.synchronize()
    n = int(cnt.item())
    return n, P.unpack_keypoints(kps[:min(n, max_kps)].cpu().numpy())


def _ordered(kp, width):
    gx = (width + 31) // 32
    k = kp.astype(np.int64)
    return kp[np.argsort(((k[:, 1] // 32) * gx + k[:, 0] // 32) * 1024 + (k[:, 1] % 32) * 32 + k[:, 0] % 32)]


def _dots(w, h, step, seed):
    """A flat image with isolated bright and dark dots of random strength: few keypoints."""
    rng = np.random.default_rng(seed)
    img = np.full((h, (w + 15) // 16 * 16), 128, np.uint8)
    ys, xs = np.meshgrid(np.arange(20, h - 20, step), np.arange(20, w - 20, step), indexing="ij")
    img[ys, xs] = rng.integers(0, 256, ys.shape)
    img[:, w:] = 0
    return img


@pytest.mark.parametrize("w, h", [(32 * 127, 32 * 129), (32 * 128, 32 * 128), (32 * 128 + 1, 32 * 128), (32 * 257, 32 * 65)])
def test_scan_passes(gpu_ctx, w, h):
    img = _dots(w, h, 97, w)
    want = _ordered(oracle.detect(img, w, h, 30), w)
    n, got = _detect(gpu_ctx, img, w, h, 30, len(want) + 16)
    assert n == len(want) and np.array_equal(got[:, :2], want[:, :2])
    gpu_ctx.check()


@pytest.mark.parametrize("kind, t", [("noise", 1), ("noise", 120), ("flat", 1), ("checker", 10)])
def test_candidate_extremes(gpu_ctx, kind, t):
    w, h = 200, 170
    rng = np.random.default_rng(3)
    img = np.zeros((h, 208), np.uint8)
    if kind == "noise":
        img[:, :w] = rng.integers(0, 256, (h, w))
    elif kind == "checker":
        img[:, :w] = 255 * ((np.add.outer(np.arange(h) // 5, np.arange(w) // 5)) & 1)
    else:
        img[:, :w] = 77
    want = _ordered(oracle.detect(img, w, h, t), w)
    n, got = _detect(gpu_ctx, img, w, h, t, w * h)
    assert n == len(want) and np.array_equal(got[:, :3], want[:, :3])
    gpu_ctx.check()


def test_angles_near_the_boundaries(gpu_ctx):
    """Two dots 10 pixels from an isolated corner pull its centroid to within 0.01 of a
    half-integer of the bin scale for some strengths: all strengths are taken."""
    w, h, step = 1664, 1664, 64
    rng = np.random.default_rng(9)
    img = np.zeros((h, w), np.uint8)
    for y in range(32, h - 32, step):
        for x in range(32, w - 32, step):
            img[y, x] = 255
            for _ in range(2):
                a, r = rng.uniform(0, 2 * np.pi), rng.uniform(7, 13)
                img[y + int(round(r * np.sin(a))), x + int(round(r * np.cos(a)))] = rng.integers(1, 30)
    want = _ordered(oracle.detect(img, w, h, 40), w)
    n, got = _detect(gpu_ctx, img, w, h, 40, len(want) + 16)
    assert n == len(want) > 500 and np.array_equal(got[:, :3], want[:, :3])
