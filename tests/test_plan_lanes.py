"""The tensor-core tiles' lanes, sign patterns and units on the CPU (csrc/plan.cpp
built with g++ by tests/plan_lanes_check.cpp from the oracle's triangle counts):
every row of a tile on exactly one lane with its own fields, lanes without a row
reading staged fields, warps of one sign pattern, and every x chunk of a tile one
unit, for long and short chunks."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from paper_2405_14513_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan_lanes")
    exe = str(d / "plan_lanes_check")
    src = os.path.join(ROOT, "paper_2405_14513_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", src,
                    os.path.join(ROOT, "tests", "plan_lanes_check.cpp"), os.path.join(src, "plan.cpp"), "-o", exe,
                    "-lpthread"], check=True)
    return d, exe


# the smallest grid, a 3 x 2^k one, one k1 bin, and tiles with full lanes
@pytest.mark.parametrize("ng,L,nk1", [(8, 100.0, 1), (24, 300.0, 3), (48, 800.0, 1), (64, 1000.0, 6)])
def test_lanes_and_units(driver, ng, L, nk1):
    d, exe = driver
    ntri, _ = O.ntri(ng)
    ntri.astype(np.int64).tofile(str(d / "ntri.bin"))
    np.asarray(synth.default_k1_edges(ng, L, nk1), dtype=np.float64).tofile(str(d / "edges.bin"))
    r = subprocess.run([exe, str(ng), repr(L), str(nk1), "5", str(d / "ntri.bin"), str(d / "edges.bin")], check=True,
                       capture_output=True, text=True)
    tiles, mixed, bad = map(int, r.stdout.split())
    assert bad == 0, r.stderr[:2000]
    assert tiles > 0
    if ng == 64:
        assert mixed > 0            # sign patterns shared some tiles
