"""The triplet list of the extraction's evaluators, made on the host for any table: every
triplet once, its patches from the quarter's part of the window or from the staged one, and
the work spread over the four quarters (each is one SM partition) also for tables whose patches
lie far apart."""
import ctypes
import time

import numpy as np
import pytest

from paper_1609_03986_gb300 import build, synth

BITS, CLASSES, STAGED = 512, 9, 8
# first byte column, word columns, first row, rows of what each quarter holds of a window
QUARTERS = [(0, 12, 0, 42), (1, 12, 6, 42), (2, 10, 0, 48), (7, 10, 0, 48)]
WINDOW = (0, 12, 0, 48)
LAST_COLUMN = 512 - 8
TABLES = ["seeded", "uniform", "centre", "one_phase", "last_rows", "last_columns", "wide", "diagonal", "corners"]


class Plan(ctypes.Structure):
    _fields_ = [("e", (ctypes.c_uint32 * BITS) * 3), ("start", (ctypes.c_int16 * (CLASSES + 1)) * 4)]


@pytest.fixture(scope="module")
def plan_triplets():
    f = ctypes.CDLL(build.build())._ZN5latch13plan_tripletsEPK13latch_tripletiPNS_15LaneTripletPlanE
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p], None
    return f


def table(kind, size):
    hi = 44 if size == 7 else 43
    rng = np.random.default_rng(5)
    t = rng.integers(3, hi + 1, (BITS, 6))
    if kind == "seeded":
        t = np.asarray(synth.triplets(lo=3, hi=hi))
    elif kind == "centre":
        t = np.clip(np.rint(rng.normal(23.5, 9, (BITS, 6))), 3, hi)
    elif kind == "one_phase":
        t[:, 0::2] = 3 + 4 * rng.integers(0, 10, (BITS, 3))
    elif kind == "last_rows":
        t[:, 1::2] = rng.integers(hi - 6, hi + 1, (BITS, 3))
    elif kind == "last_columns":
        t[:, 0::2] = rng.integers(hi - 6, hi + 1, (BITS, 3))
    elif kind == "wide":
        t[:, 0], t[:, 2] = rng.integers(3, 8, BITS), rng.integers(hi - 4, hi + 1, BITS)
    elif kind == "diagonal":
        t[:, 0:2], t[:, 2:4] = rng.integers(3, 9, (BITS, 2)), rng.integers(hi - 5, hi + 1, (BITS, 2))
    elif kind == "corners":
        t = rng.choice([3, hi], (BITS, 6))
    return np.ascontiguousarray(t, dtype=np.uint8)


@pytest.mark.parametrize("size", [7, 8])
@pytest.mark.parametrize("kind", TABLES)
def test_plan(plan_triplets, kind, size):
    t, plan = table(kind, size), Plan()
    plan_triplets(t.ctypes.data, size, ctypes.byref(plan))
    e = np.array(plan.e, dtype=np.int64)
    start = np.array(plan.start)
    assert start[0, 0] == 0 and start[3, CLASSES] == BITS
    assert (start[1:, 0] == start[:-1, CLASSES]).all() and (np.diff(start, axis=1) >= 0).all()
    assert sorted((e[0] >> 5) & 511) == list(range(BITS))
    for q in range(4):
        for cls in range(CLASSES):
            b0, nc, r0, nr = WINDOW if cls == STAGED else QUARTERS[q]
            for at in range(start[q, cls], start[q, cls + 1]):
                patches = t[(e[0, at] >> 5) & 511].astype(int).reshape(3, 2) - 3
                for p, (x0, y0) in enumerate(patches):
                    x, y = x0 - b0, y0 - r0
                    assert 0 <= x <= 4 * nc - size and 0 <= y <= nr - size
                    assert e[p, at] >> 16 == (x >> 2) * nr + y and (e[p, at] & 31) == 8 * (x & 3)
                    if cls != STAGED:
                        assert ((cls >> p) & 1) == int((x & 3) != 0)
                        assert (x & 3) == 0 or ((x >> 2) + 2) * nr + y <= LAST_COLUMN
    # a quarter is one SM partition: none may take more than half of the triplets
    assert (start[:, CLASSES] - start[:, 0]).max() <= BITS // 2


@pytest.mark.parametrize("size", [7, 8])
@pytest.mark.parametrize("kind", ["seeded", "uniform", "last_rows"])
def test_plan_is_quick(plan_triplets, kind, size):
    """An extraction that is given another table than the last one plans it first: that has
    to stay small next to a launch (best of many runs; searching the table for every move took 0.2 ms and more)."""
    t, plan, best = table(kind, size), Plan(), 1.0
    for _ in range(50):
        t0 = time.perf_counter()
        plan_triplets(t.ctypes.data, size, ctypes.byref(plan))
        best = min(best, time.perf_counter() - t0)
    assert best < 1.5e-4
