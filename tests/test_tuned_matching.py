"""What the autotuner keeps of its matching ladder: the pair threshold, and the rule that sends
smaller problems to the tensor cores unless a rung of the rule's range was measured the other
way.  A threshold of 2^22 stands for the default, so a measured one without the rule is never
exactly that."""
import ctypes

import pytest

from paper_1609_03986_gb300 import build

DEFAULT = 1 << 22


class Rung(ctypes.Structure):
    _fields_ = [("nt", ctypes.c_int64), ("tensor_wins", ctypes.c_bool)]


@pytest.fixture(scope="module")
def tuned():
    f = ctypes.CDLL(build.build())._ZN5latch14tuned_matchingElPKNS_9MatchRungEiPlPb
    f.restype = None

    def run(nq, rungs):
        pairs, small = ctypes.c_int64(), ctypes.c_bool()
        f(ctypes.c_int64(nq), (Rung * len(rungs))(*rungs), len(rungs), ctypes.byref(pairs), ctypes.byref(small))
        return pairs.value, small.value
    return run


@pytest.mark.parametrize("nq, rungs, pairs, small", [
    # the tensor path wins from the first rung of the rule's range on, or earlier
    (10000, [(64, False), (256, True)], 2560000, True),
    (10000, [(64, False), (256, False), (1024, True)], 10240000, True),
    (300, [(64, True)], 19200, True),
    # no rung of the range was measured
    (16384, [(64, False)], DEFAULT, True),
    (1, [(64, False), (256, False)], 1024, True),
    # the CUDA cores win in the range: a plain threshold
    (100, [(64, False), (256, False), (1024, False), (4096, True)], 409600, False),
    (2000, [(64, False), (256, False), (1024, False), (2000, False)], 16000000, False),
    # the same where the threshold would be the default value
    (1024, [(64, False), (256, False), (1024, False)], DEFAULT + 1, False),
    (1024, [(64, False), (256, False), (1024, False), (4096, True)], DEFAULT - 1, False),
    # few queries against 17,000 to 30,000 rows are not in the range
    (8, [(64, False), (256, False), (20000, False)], 640000, True),
])
def test_what_is_kept(tuned, nq, rungs, pairs, small):
    assert tuned(nq, rungs) == (pairs, small)
