"""Changing the scale table between host-memory batches: the batch's device staging sets
and upload stream outlive latch_set_scales."""
import numpy as np
import pytest
import torch

import paper_1609_03986_gb300 as P
from paper_1609_03986_gb300 import synth

pytestmark = pytest.mark.gpu

W, H, N = 320, 240, 300


def _pinned(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy()).pin_memory()


def test_set_scales_between_host_batches(triplets):
    ctx = P.Context(0, triplets=triplets)
    img = synth.image(synth.seed(71, 0, synth.KIND_IMAGE), W, H, n_ellipses=20)
    kps = P.pack_keypoints(synth.keypoints(synth.seed(71, 0, synth.KIND_KEYPOINTS), W, H, N, 0, True, 3))
    d_img, d_kps = torch.from_numpy(img).cuda(), torch.from_numpy(kps).cuda()
    h_img, h_kps = _pinned(img), _pinned(kps)
    stream = torch.cuda.current_stream()
    for scales in ((1.0, 1.5, 2.25), (1.0, 1.25, 2.0), (1.0, 1.5, 2.25)):
        P.latch_set_scales(ctx.handle, scales)
        for _ in range(2):  # both staging sets
            h_desc = torch.zeros(N * 64, dtype=torch.uint8, pin_memory=True)
            h_m = torch.zeros(N * 16, dtype=torch.uint8, pin_memory=True)
            hb = P.HostBatchDesc([(h_img, W, H, img.shape[1])], [N], h_kps, h_desc, [(0, 0)], 2, 0.8, h_m)
            P.latch_batch_run_host(ctx.handle, hb, int(stream.cuda_stream))
            torch.cuda.synchronize()
            want = ctx.extract(d_img, W, H, d_kps)
            torch.cuda.synchronize()
            assert np.array_equal(h_desc.numpy().reshape(N, 64), want.cpu().numpy())
    ctx.check()
