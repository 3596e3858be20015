"""The windowed integer sum of gf_winsum.cuh built for the host, filled to the
last term between two folds with the largest values its window takes."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_full_window_does_not_overflow(tmp_path):
    exe = str(tmp_path / "winsum_limit_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2306_11686_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "winsum_limit_check.cpp"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300).stdout
    m = re.search(r"sums checked (\d+) mismatches (\d+)", out)
    assert m and int(m.group(1)) == 320 and int(m.group(2)) == 0, out
