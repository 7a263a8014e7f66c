"""The x chunk length of a tensor-core plan, set after the enumeration, on the CPU
(csrc/plan.cpp built with g++ by tests/plan_chunk_check.cpp from the oracle's triangle
counts): the same plan as one enumerated for that length."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from paper_2405_14513_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


# the smallest grid, one that is not of 2^k, and one whose largest grids take several chunks
@pytest.mark.parametrize("ng,L,nk1", [(8, 100.0, 1), (48, 800.0, 3), (64, 1000.0, 6)])
def test_x_chunk_set_afterwards(tmp_path, ng, L, nk1):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "plan_chunk_check")
    src = os.path.join(ROOT, "paper_2405_14513_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", src,
                    os.path.join(ROOT, "tests", "plan_chunk_check.cpp"), os.path.join(src, "plan.cpp"), "-o", exe,
                    "-lpthread"], check=True)
    ntri, _ = O.ntri(ng)
    ntri.astype(np.int64).tofile(str(tmp_path / "ntri.bin"))
    np.asarray(synth.default_k1_edges(ng, L, nk1), dtype=np.float64).tofile(str(tmp_path / "edges.bin"))
    r = subprocess.run([exe, str(ng), repr(L), str(nk1), str(tmp_path / "ntri.bin"), str(tmp_path / "edges.bin")], check=True,
                       capture_output=True, text=True)
    units, bad = map(int, r.stdout.split())
    assert units > 0 and bad == 0
