"""The tensor matcher at the edges of its tiles: 256 queries per block pair (128 in each
block), 240 train rows per unit (120 from each block's shared memory), and the split of the
units over the pairs.  Exact: every field of every record against the oracle (small sizes)
or the CUDA-core path (larger ones)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_03986_gb300 as P
from paper_1609_03986_gb300 import synth

pytestmark = pytest.mark.gpu

FIELDS = ("idx1", "idx2", "dist1", "dist2", "accepted")


def _sets(nq, nt, salt):
    q = synth.random_descriptors(synth.seed(71, 2 * salt, synth.KIND_GALLERY), nq)
    t = synth.random_descriptors(synth.seed(71, 2 * salt + 1, synth.KIND_GALLERY), nt)
    t[::5] = q[0]          # ties over the whole train set
    t[-1] = q[-1]          # an exact match in the last row
    return q, t


def _run(ctx, q, t, k, path):
    out = ctx.match(torch.from_numpy(q).cuda(), torch.from_numpy(t).cuda(), k, 0.8, path)
    return P.matches_from_bytes(out.cpu().numpy())


@pytest.mark.parametrize("nq", [1, 127, 128, 129, 255, 256, 257])
@pytest.mark.parametrize("nt", [1, 119, 120, 121, 239, 240, 241, 479, 481])
def test_tile_edges(gpu_ctx, nq, nt):
    q, t = _sets(nq, nt, nq * 1000 + nt)
    for k in (1, 2):
        got, want = _run(gpu_ctx, q, t, k, P.PATH_TENSOR), oracle.match(q, t, k, 0.8)
        for f in FIELDS:
            assert np.array_equal(got[f].astype(np.int64), np.asarray(want[f]).astype(np.int64)), (k, f)
    gpu_ctx.check()


@pytest.mark.parametrize("nq, nt", [(256 * 19, 240 * 4), (256 * 19 + 1, 240 * 4 + 1), (300, 240 * 76), (300, 240 * 76 + 7),
                                    (20000, 241), (5000, 31000), (513, 100003)])
def test_splits_over_the_pairs(gpu_ctx, nq, nt):
    """One unit per pair, one more, many tiles of one unit, and walks that end inside a
    tile, in short (combined in the launch) and long launches."""
    q, t = _sets(nq, nt, nq + nt)
    got, want = (_run(gpu_ctx, q, t, 2, p) for p in (P.PATH_TENSOR, P.PATH_POPC))
    for f in FIELDS:
        assert np.array_equal(got[f], want[f]), f
    gpu_ctx.check()


@pytest.mark.parametrize("nq", [1, 17, 300, 2000])
@pytest.mark.parametrize("nt", [1, 255, 256, 257, 2000])
def test_auto_route(gpu_ctx, nq, nt):
    """LATCH_PATH_AUTO below its pair threshold: the CUDA cores up to 256 train rows, the
    tensor cores beyond (the threshold alone once it is set), the same records on both."""
    want = P.PATH_TENSOR if nt > 256 else P.PATH_POPC
    assert P.hamming_match_path(gpu_ctx.handle, nq, nt) == want
    q, t = _sets(nq, nt, nq + 3 * nt)
    for k in (1, 2):
        got, ref = _run(gpu_ctx, q, t, k, P.PATH_AUTO), _run(gpu_ctx, q, t, k, P.PATH_POPC)
        for f in FIELDS:
            assert np.array_equal(got[f], ref[f]), (k, f)
    saved = P.latch_get_tuning(gpu_ctx.handle)
    try:
        P.latch_set_tuning(gpu_ctx.handle, saved["item_kps"], saved["tensor_min_pairs"] + 1)
        assert P.hamming_match_path(gpu_ctx.handle, nq, nt) == P.PATH_POPC
    finally:
        P.latch_set_tuning(gpu_ctx.handle, saved["item_kps"], saved["tensor_min_pairs"])
