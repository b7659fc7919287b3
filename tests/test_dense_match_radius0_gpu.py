"""Windowed matching at radius 0, where each pixel has itself as its only candidate and nothing
is staged: at the edges of the 16x16-pixel tiles, both k."""
import numpy as np
import pytest
import torch

import oracle
from conftest import match_records, same_matches, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(1, 1), (15, 17), (16, 16), (33, 5), (1, 40), (257, 31)])
@pytest.mark.parametrize("k", [1, 2])
def test_radius_zero(gpu_ctx, w, h, k):
    rng = np.random.default_rng(w + 100 * h)
    da, db = (rng.integers(0, 256, (w * h, 64), dtype=np.uint8) for _ in range(2))
    da[::3] = db[::3]
    out = gpu_ctx.dense_match(to_dev(da), to_dev(db), w, h, 0, k, 0.8)
    torch.cuda.synchronize()
    same_matches(match_records(out), oracle.dense_match(da, db, w, h, 0, k, 0.8))
    gpu_ctx.check()
