"""The highest window of gf_fixsum.cuh, built for the host: its sums of six
are IEEE's bit for bit, and one binade higher they are not (there the IEEE sum
overflows and the chunks' does not)."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_highest_window_is_the_last_without_overflow(tmp_path):
    exe = str(tmp_path / "fixsum_top_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-frounding-math", "-I",
                    os.path.join(ROOT, "paper_2306_11686_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "fixsum_top_check.cpp"), "-o", exe],
                   check=True, capture_output=True)

    def run(top):
        out = subprocess.run([exe, str(top)], capture_output=True, text=True, timeout=300).stdout
        m = re.search(r"div6 checked 200000 mismatches (\d+), highest window (\d+)", out)
        assert m, out
        return int(m.group(1)), int(m.group(2))

    top = run(1023)[1]
    assert run(1023)[0] == 0 and run(top - 1)[0] == 0
    assert run(top)[0] == 0
    assert run(top + 1)[0] > 0
