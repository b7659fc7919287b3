"""Single problems whose query tiles are walked by several block pairs that exchange row
bounds: matches equal the CUDA-core path's, with ties at every distance and with rows whose
two best lie in different pairs' parts of the train set."""
import numpy as np
import pytest
import torch

import paper_1609_03986_gb300 as P
from conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,nt,pool", [(1, 60001, 40), (257, 20011, 0), (300, 17000, 3), (1300, 40000, 200),
                                        (2340, 30000, 0), (9985, 5000, 64)])
def test_shared_bounds_exact(gpu_ctx, nq, nt, pool):
    rng = np.random.default_rng(nq + nt)
    q = rng.integers(0, 256, (nq, 64), dtype=np.uint8)
    if pool:  # few train values: every distance is tied many times, far apart
        t = rng.integers(0, 256, (pool, 64), dtype=np.uint8)[rng.integers(0, pool, nt)]
    else:  # each query's best at the end of the train set, its second best at the start
        t = rng.integers(0, 256, (nt, 64), dtype=np.uint8)
        t[nt - nq:] = q
        t[:nq] = q
        t[:nq, 0] ^= 1
    got = [gpu_ctx.match(to_dev(q), to_dev(t), 2, 0.8, path) for path in (P.PATH_TENSOR, P.PATH_POPC)]
    torch.cuda.synchronize()
    gpu_ctx.check()
    assert torch.equal(got[0], got[1])
