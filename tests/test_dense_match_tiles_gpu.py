"""Windowed matching at the edges of its 16x16-pixel tiles and of its groups of eight
staged descriptors (a radius of odd parity leaves the last group half filled)."""
import numpy as np
import pytest
import torch

import oracle
from conftest import match_records, same_matches, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,radius,k", [(1, 1, 16, 2), (16, 16, 3, 2), (17, 33, 5, 2), (50, 1, 8, 1),
                                          (1, 40, 15, 2), (35, 31, 16, 2)])
def test_dense_match_tile_edges(gpu_ctx, w, h, radius, k):
    rng = np.random.default_rng(7 * w + h)
    pool = rng.integers(0, 256, (6, 64), dtype=np.uint8)  # few values: ties in every window
    da, db = (pool[rng.integers(0, 6, w * h)] for _ in range(2))
    out = gpu_ctx.dense_match(to_dev(da), to_dev(db), w, h, radius, k, 0.8)
    torch.cuda.synchronize()
    same_matches(match_records(out), oracle.dense_match(da, db, w, h, radius, k, 0.8))
