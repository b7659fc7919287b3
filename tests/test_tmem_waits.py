"""Registers written by an asynchronous tensor-memory load are undefined until the wait, and
the wait names none of them: behind every wait the loaded registers are tied to it at once
(or nothing reads them any more), so that no arithmetic on them can be moved above it."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# the statement behind the wait: a tie of loaded registers, possibly in an unrolled loop, or
# the end of the function
TIED = re.compile(r"\s*(#pragma unroll\s+)?(for \([^{};]*;[^{};]*;[^{};]*\)\s*)?(arrive<|tmem_arrived\(|\})")


def test_every_load_wait_ties_its_registers():
    waits = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1609_03986_gb300", "csrc", "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\btmem_ld_wait\(\);", src):
            waits += 1
            line = src.count("\n", 0, m.start()) + 1
            assert TIED.match(src, m.end()), f"{os.path.basename(path)}:{line}: loaded registers used without a tie"
    assert waits >= 2  # the extraction's and the matcher's
