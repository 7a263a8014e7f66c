"""Blocks of the binning's last pass (fin_bins_per_block of csrc/plan.hpp) on the CPU:
within a launch's limits for any number of bins that a plan can have, one bin each
where bins are few."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <cstdio>
#include "plan.hpp"
int main()
{
    for (long long n; std::scanf("%lld", &n) == 1;) std::printf("%lld\\n", (long long)bisp::fin_bins_per_block(n));
}
"""


def test_fin_blocks(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    (tmp_path / "f.cpp").write_text(SRC)
    exe = str(tmp_path / "f")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2405_14513_gb300", "csrc"), str(tmp_path / "f.cpp"), "-o", exe], check=True)
    sizes = [1, 2, 12000, 16384, 16385, 32768, 32769, 1200000, 2 ** 31 - 1, 2 ** 31, 5 * 2 ** 31]
    r = subprocess.run([exe], input="\n".join(map(str, sizes)), capture_output=True, text=True, check=True)
    for n, per in zip(sizes, map(int, r.stdout.split())):
        assert per >= 1 and -(-n // per) <= 16384, (n, per)
        assert (per == 1) == (n <= 16384), (n, per)
