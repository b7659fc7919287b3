"""Orientations on the bin boundaries.  The detection takes the angle in FP32 and computes it
again in FP64 where it lies within 1e-3 of a boundary; these moments lie so close to one that
FP32 alone gives another bin for many of them, and just outside that window, on both sides of
every boundary."""
import numpy as np
import pytest

import oracle

STEP, T, MOMENT = 64, 40, 4000
W = H = 46 * STEP


def _position(m10, m01):
    """The angle on the bin scale, FP64."""
    return np.arctan2(np.float64(m01), np.float64(m10)) * 16 / np.pi


def _from_boundary(p):
    return np.abs(np.abs(p - np.round(p)) - 0.5)


def _moments():
    """(m10, m01) next to the 32 boundaries: the closest ones on each side among moments up
    to MOMENT, and some just inside and outside of 1e-3."""
    out = []
    a = np.arange(60, MOMENT)
    for k in range(4):  # boundaries below 45 degrees; the others by exchange and sign
        b = np.rint(a * np.tan((k + 0.5) * np.pi / 16)).astype(int)
        off = _position(a, b) - (k + 0.5)
        ok = (b >= 5) & (np.gcd(a, b) == 1)
        picks = []
        for side in (off > 0, off < 0):
            idx = np.flatnonzero(ok & side)
            picks += list(idx[np.argsort(np.abs(off[idx]))[:24]])
            picks += list(idx[np.argsort(np.abs(np.abs(off[idx]) - 1e-3))[:8]])
        for i in picks:
            x, y = int(a[i]), int(b[i])
            out += [(sx * u, sy * v) for u, v in ((x, y), (y, x)) for sx in (1, -1) for sy in (1, -1)]
    return out


def _split(m, d=15):
    """m >= 0 as a sum of value * distance, distances d down to 5, values below the threshold."""
    if m == 0:
        return []
    if d < 5:
        return None
    most = min(T - 1, m // d)
    for v in range(most, max(most - 3, 0) - 1, -1):
        rest = _split(m - v * d, d - 1)
        if rest is not None:
            return ([(d, v)] if v else []) + rest
    return None


def _dots(m):
    return [(d if m > 0 else -d, v) for d, v in _split(abs(m))]


def _scene():
    img = np.zeros((H, W), np.uint8)
    moments = _moments()
    n = W // STEP
    assert len(moments) <= n * n
    for i, (m10, m01) in enumerate(moments):
        x, y = STEP // 2 + STEP * (i % n), STEP // 2 + STEP * (i // n)
        img[y, x] = 255
        for d, v in _dots(m10):
            img[y, x + d] = v
        for d, v in _dots(m01):
            img[y + d, x] = v
    return img, np.array(moments)


def _bins(p):
    return (np.floor(np.abs(p) + 0.5) * np.sign(p)).astype(int) % 32


def test_fp32_alone_gives_other_bins():
    """The scene is one that an angle in FP32 gets wrong (numpy's arctan2, rounded like the
    kernel's), and the oracle's bins are the FP64 ones."""
    img, m = _scene()
    p = _position(m[:, 0], m[:, 1])
    near = _from_boundary(p)
    assert (near < 1e-3).sum() > 500 and (near < 1e-6).sum() > 50 and ((near >= 1e-3) & (near < 2e-3)).sum() > 100
    single = np.arctan2(m[:, 1].astype(np.float32), m[:, 0].astype(np.float32)) * np.float32(16 / np.pi)
    wrong = np.rint(single).astype(int) % 32 != _bins(p)
    assert wrong.sum() >= 8 and near[wrong].max() < 1e-5
    kp = oracle.detect(img, W, H, T)
    assert len(kp) == len(m)
    order = np.lexsort((kp[:, 0], kp[:, 1]))
    assert np.array_equal(kp[order][:, 2], _bins(p))


@pytest.mark.gpu
def test_bins_are_the_fp64_ones(gpu_ctx):
    import torch

    import paper_1609_03986_gb300 as P
    from conftest import to_dev
    img, m = _scene()
    kps, cnt = gpu_ctx.detect(to_dev(img), W, H, T, len(m) + 16)
    torch.cuda.synchronize()
    assert int(cnt.item()) == len(m)
    kp = P.unpack_keypoints(kps[:len(m)].cpu().numpy()).astype(int)
    order = np.lexsort((kp[:, 0], kp[:, 1]))
    assert np.array_equal(kp[order][:, 2], _bins(_position(m[:, 0], m[:, 1])))
    gpu_ctx.check()
