"""LATCH_PATH_AUTO after tuning: an autotuned context still sends small problems to the tensor
cores (on which they are measured faster), a threshold set by hand is a plain threshold, and
the default value brings the default rule back."""
import pytest

import paper_1609_03986_gb300 as P

pytestmark = pytest.mark.gpu


def test_routes_after_tuning(triplets):
    ctx = P.Context(0, triplets=triplets)
    try:
        h = ctx.handle
        default = P.latch_get_tuning(h)["tensor_min_pairs"]
        assert default == 1 << 22 and P.hamming_match_path(h, 1000, 1000) == P.PATH_TENSOR
        t = P.latch_autotune(h, 640, 480, 0, 10000, 10000)
        assert P.hamming_match_path(h, 1000, 1000) == P.PATH_TENSOR
        P.latch_set_tuning(h, t["item_kps"], t["tensor_min_pairs"])  # its own values: nothing changes
        assert P.hamming_match_path(h, 1000, 1000) == P.PATH_TENSOR
        for value, path in ((2000000, P.PATH_POPC), (default - 1, P.PATH_POPC), (default + 1, P.PATH_POPC),
                            (default, P.PATH_TENSOR), (1000000, P.PATH_TENSOR), (default, P.PATH_TENSOR)):
            P.latch_set_tuning(h, t["item_kps"], value)
            assert P.hamming_match_path(h, 1000, 1000) == path, value
    finally:
        ctx.close()
