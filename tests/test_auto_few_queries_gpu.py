"""LATCH_PATH_AUTO with few queries: against 17,000 to 30,000 train rows up to 12 queries stay
on the CUDA cores (36,000 - 1,000 nq rows at most), around that the tensor cores take them;
the same records on both paths."""
import numpy as np
import pytest
import torch

import paper_1609_03986_gb300 as P
from conftest import to_dev

pytestmark = pytest.mark.gpu

NT = (17000, 17001, 23999, 24001, 28000, 28001, 30000, 30001, 65536, 65537)


@pytest.fixture(scope="module")
def train():
    t = np.random.default_rng(3).integers(0, 256, (max(NT), 64), dtype=np.uint8)
    t[::97] = t[5]  # ties all over the set
    return t, to_dev(t)


@pytest.mark.parametrize("nq", [1, 6, 8, 12, 13, 63])
def test_route_and_records(gpu_ctx, train, nq):
    t, d_t = train
    q = np.random.default_rng(nq).integers(0, 256, (nq, 64), dtype=np.uint8)
    q[0] = t[5]
    d_q = to_dev(q)
    for nt in NT:
        few = nq <= 12 and 17000 < nt <= min(30000, 36000 - 1000 * nq)
        want = P.PATH_POPC if few or nt > 65536 else P.PATH_TENSOR
        assert P.hamming_match_path(gpu_ctx.handle, nq, nt) == want, nt
        for k in (1, 2):
            got, a, b = (gpu_ctx.match(d_q, d_t[:nt], k, 0.8, path) for path in (P.PATH_AUTO, P.PATH_POPC, P.PATH_TENSOR))
            torch.cuda.synchronize()
            assert torch.equal(got, a) and torch.equal(a, b), (nt, k)
    gpu_ctx.check()
