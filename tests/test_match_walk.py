"""How the tensor matcher deals a launch's units out to the block pairs, walked on the host
through the kernel's own share functions: every unit exactly once, and in launches that share
whole query tiles no pair more than one tile above another (problems of equal size)."""
import os
import subprocess

import pytest

from paper_1609_03986_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("walk") / "match_walk")
    subprocess.run([os.path.join(build._cuda_home(), "bin", "nvcc"), *build.ARCH, "-std=c++17", "-O1",
                    "--expt-relaxed-constexpr", "-I" + build.INCLUDE, "-I" + build.CSRC,
                    os.path.join(ROOT, "tests", "match_walk.cu"), lib, "-Xlinker", "-rpath," + os.path.dirname(lib),
                    "-o", exe], check=True)

    def run(sms, count, *sets):
        out = subprocess.run([exe, str(sms), str(count)] + [str(v) for s in sets for v in s], check=True,
                             capture_output=True, text=True).stdout
        names = ("whole", "pairs", "most", "fewest", "walked", "distinct", "units")
        return dict(zip(names, map(int, out.split())))
    return run


@pytest.mark.parametrize("n", [60, 300, 500, 600, 1000, 1500, 2000, 2340, 3000, 5000, 10000])
@pytest.mark.parametrize("count", [476, 512])
def test_whole_tiles_are_dealt_out_evenly(walk, n, count):
    r = walk(SMS, count, (n, n))
    assert r["walked"] == r["distinct"] == r["units"]
    tile = (n + 239) // 240
    if r["whole"]:
        assert r["most"] - r["fewest"] <= tile
    else:
        assert n == 60 and count < 608


@pytest.mark.parametrize("sms", [1, 2, 3, 148, 152])
@pytest.mark.parametrize("sets", [[(2340, 2340)], [(1, 1), (0, 50), (257, 241), (4000, 0)], [(0, 9), (700, 481)],
                                  [(200000, 300)], [(5, 100003)]])
def test_every_unit_once(walk, sms, sets):
    for count in (1, 7, 131):
        r = walk(sms, count, *sets)
        assert r["walked"] == r["distinct"] == r["units"]
