"""Parity of the extraction's batches, tile classes and triplet plan at the sizes where they
change (exact bytes; the descriptors are integers, so the tolerance is equality).

The launch takes keypoints in batches of up to 32, whole batches in rounds over the
blocks and the last round cut into chunk ranges; a scale table is served by at most three
tile boxes; a triplet table is planned over four tensor-memory quarters, and what fits
none of them takes rows from shared memory."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_03986_gb300 as P
from paper_1609_03986_gb300 import synth

pytestmark = pytest.mark.gpu

W, H = 520, 400


def _image():
    return synth.image(synth.seed(61, 0, synth.KIND_IMAGE), W, H, n_ellipses=40)


def _extract(ctx, img, kps):
    return ctx.extract(torch.from_numpy(img).cuda(), W, H, torch.from_numpy(P.pack_keypoints(kps)).cuda()).cpu().numpy()


@pytest.fixture(scope="module")
def many():
    """Keypoints for three rounds of any launch, some of them outside the image."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 3 * 32 * sms
    rng = np.random.default_rng(61)
    kps = np.stack([rng.integers(-60, W + 60, n), rng.integers(-60, H + 60, n), rng.integers(0, 32, n),
                    rng.integers(0, 3, n)], 1).astype(np.int32)
    return sms, kps


@pytest.mark.parametrize("rounds, extra", [(1, -1), (1, 0), (1, 1), (1, 33), (2, -40), (2, 0), (2, 31), (3, 0)])
def test_rounds_equal_small_launches(gpu_ctx, triplets, many, rounds, extra):
    """Around whole rounds of 32 keypoints per block: every row equals the row of a launch
    of 97 keypoints (a single incomplete round), and the last rows and a seeded sample
    equal the oracle."""
    sms, kps = many
    n = rounds * 32 * sms + extra
    img = _image()
    got = _extract(gpu_ctx, img, kps[:n])
    rows = np.unique(np.concatenate([np.arange(n - 8, n), np.random.default_rng(n).integers(0, n, 16)]))
    assert np.array_equal(got[rows], oracle.extract(img, W, H, kps[rows], triplets, synth.SCALES))
    for r0 in (0, min(32 * sms - 48, n - 97), n - 97):
        assert np.array_equal(got[r0:r0 + 97], _extract(gpu_ctx, img, kps[r0:r0 + 97])), r0
    gpu_ctx.check()


@pytest.mark.parametrize("scales", [(0.25,), (2.25,), (0.3, 0.5, 0.75, 1.0, 1.3, 1.6, 1.9, 2.25), (1.0, 1.0, 2.0, 2.0)])
def test_tile_classes_of_scale_tables(triplets, scales):
    """Scale tables of one, a few and eight scales (several scales share a tile box)."""
    ctx = P.Context(0, scales=scales, triplets=triplets)
    try:
        img = _image()
        rng = np.random.default_rng(len(scales))
        n = 6 * len(scales) + 32
        kps = np.stack([rng.integers(-20, W + 20, n), rng.integers(-20, H + 20, n), np.arange(n) % 32,
                        np.arange(n) % len(scales)], 1).astype(np.int32)
        assert np.array_equal(_extract(ctx, img, kps), oracle.extract(img, W, H, kps, triplets, scales))
        ctx.check()
    finally:
        ctx.close()


@pytest.mark.parametrize("kind", ["corners", "last_rows", "last_columns", "one_phase", "wide"])
@pytest.mark.parametrize("weighted", [False, True])
def test_triplet_plans(kind, weighted):
    """Triplet tables that crowd one quarter: patches in all corners (no quarter holds them),
    in the last rows or word columns, all starting at the same byte of a word, and
    triplets as wide as the window."""
    hi = 43 if weighted else 44
    rng = np.random.default_rng(5)
    t = rng.integers(3, hi + 1, (512, 6))
    if kind == "corners":
        t = rng.choice([3, hi], (512, 6))
    elif kind == "last_rows":
        t[:, 1::2] = rng.integers(hi - 6, hi + 1, (512, 3))
    elif kind == "last_columns":
        t[:, 0::2] = rng.integers(hi - 6, hi + 1, (512, 3))
    elif kind == "one_phase":
        t[:, 0::2] = 3 + 4 * rng.integers(0, 10, (512, 3))
    else:
        t[:, 0], t[:, 2] = rng.integers(3, 8, 512), rng.integers(hi - 4, hi + 1, 512)
    t = t.astype(np.uint8)
    weights = rng.integers(0, 256, (8, 8)).astype(np.uint8) if weighted else None
    ctx = P.Context(0, triplets=t)
    try:
        if weighted:
            P.latch_set_patch_weights(ctx.handle, weights)
        img = _image()
        n = 40
        kps = np.stack([rng.integers(0, W, n), rng.integers(0, H, n), rng.integers(0, 32, n), rng.integers(0, 3, n)],
                       1).astype(np.int32)
        assert np.array_equal(_extract(ctx, img, kps), oracle.extract(img, W, H, kps, t, synth.SCALES, weights=weights))
        if weighted:  # back to plain patches: the plan is made again for 7 x 7
            P.latch_set_patch_weights(ctx.handle, None)
            assert np.array_equal(_extract(ctx, img, kps), oracle.extract(img, W, H, kps, t, synth.SCALES))
        ctx.check()
    finally:
        ctx.close()
