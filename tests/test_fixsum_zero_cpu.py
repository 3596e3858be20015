"""Sums of zeros in gf_fixsum.cuh, built for the host."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_sum_of_zeros_is_accepted(tmp_path):
    exe = str(tmp_path / "fixsum_zero_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-frounding-math", "-I",
                    os.path.join(ROOT, "paper_2306_11686_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "fixsum_zero_check.cpp"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300).stdout
    m = re.search(r"zero checked (\d+) mismatches (\d+)", out)
    assert m and int(m.group(1)) == 7 * (2035 - 5 + 1) and int(m.group(2)) == 0, out
