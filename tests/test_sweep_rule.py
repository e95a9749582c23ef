"""CPU check of the rule that sets the CTAs per SM of the exact level's sweep
update (csrc/sweep_rule.h): two in the first wave of three per SM beyond two CTAs per
SM and in three fifths of the second, three otherwise."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_21618_gb300", "csrc")
MAIN = """
#include <stdio.h>
#include "sweep_rule.h"
int main() { for (int t = 0; t <= 2000; ++t) putchar(slrf::sweep_three_per_sm(152, t) ? '3' : '2'); }
"""


def test_ctas_per_sm(tmp_path):
    gxx = shutil.which(os.environ.get("CXX", "g++"))
    if gxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rule.cpp", str(tmp_path / "rule")
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I" + CSRC, str(src), "-o", exe], check=True)
    got = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    wave = 3 * 152
    for t, g in enumerate(got):
        assert g == ("2" if 2 * 152 < t <= 1.6 * wave else "3"), t
    measured = {112: "3", 264: "3", 420: "2", 480: "2", 684: "2", 760: "3", 840: "3", 912: "3", 918: "3", 1104: "3",
                1224: "3", 1368: "3"}
    for t, want in measured.items():
        assert got[t] == want
