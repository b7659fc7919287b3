"""Two requests in one micro-batch of a session, with query counts at the edges of the tensor
matcher's tiles (128 query rows in each block of a pair, 256 together) and galleries at those of
its 240-row units: the same records as a call of its own on the CUDA cores."""
import time

import numpy as np
import pytest
import torch

import paper_1609_03986_gb300 as P
from paper_1609_03986_gb300 import synth
from conftest import to_dev

pytestmark = pytest.mark.gpu

W, H = 640, 480
GALLERIES = (239, 240, 241, 2500)
COUNTS = (127, 128, 129, 255, 256, 257)


@pytest.fixture(scope="module")
def serving(triplets):
    sess = P.Session(triplets, hbm_budget=1 << 30, max_gallery_rows=1 << 14, max_batch=8, max_batch_kps=1 << 15, lanes=1)
    gals = [synth.random_descriptors(synth.seed(52, g, synth.KIND_GALLERY), n) for g, n in enumerate(GALLERIES)]
    for g in gals:
        sess.add_gallery(g)
    img = synth.image(synth.seed(52, 0, synth.KIND_IMAGE), W, H, n_ellipses=40)
    yield sess, gals, img
    sess.close()


class _Request:
    def __init__(self, img, n, gallery, seed):
        self.img = P.pinned_copy(img)
        self.kps = P.pinned_copy(P.pack_keypoints(synth.keypoints(synth.seed(52, seed, synth.KIND_KEYPOINTS), W, H, n, 0,
                                                                  True, 3)))
        self.matches = P.pinned_copy(np.zeros((n, 16), np.uint8))
        self.n, self.gallery = n, gallery
        self.req = P.latch_request(self.img.ctypes.data, W, H, self.img.strides[0], self.kps.ctypes.data, n, gallery, 2,
                                   0.8, self.matches.ctypes.data, 0)


@pytest.mark.parametrize("first", COUNTS)
@pytest.mark.parametrize("second", COUNTS)
def test_pairs_in_a_micro_batch(serving, gpu_ctx, first, second):
    sess, gals, img = serving
    plug = _Request(img, 8000, 3, 1)
    pair = [_Request(img, first, (first + second) % 4, 2), _Request(img, second, first % 4, 3)]
    for attempt in range(60):  # until both are taken together, behind the first request or with it
        tickets = [P.latch_submit(sess.handle, plug.req)]
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 1e-5 * (attempt % 20):  # the scheduler wakes up some time after it
            pass
        tickets += [P.latch_submit(sess.handle, r.req) for r in pair]
        sizes = [P.latch_wait(sess.handle, t).batch_size for t in tickets]
        for t in tickets:
            P.latch_release(sess.handle, t)
        if sizes in ([1, 2, 2], [3, 3, 3]):
            break
    else:
        pytest.fail("the two requests never shared a micro-batch")
    for r in pair:
        d = gpu_ctx.extract(to_dev(img), W, H, to_dev(np.array(r.kps)))
        want = gpu_ctx.match(d, to_dev(gals[r.gallery]), 2, 0.8, P.PATH_POPC)
        torch.cuda.synchronize()
        assert np.array_equal(r.matches, want.cpu().numpy())
