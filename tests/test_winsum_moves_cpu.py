"""Values that no window of gf_winsum.cuh holds cost a warp about what the
compensated FP64 sum alone costs, one addition a value, and values that drift
take their window along."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_windows_do_not_move_to_and_fro(tmp_path):
    exe = str(tmp_path / "winsum_moves_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2306_11686_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "winsum_moves_check.cpp"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300).stdout
    cost = {k: int(a) / int(s) for k, a, s in re.findall(r"(\w+) adds (\d+) steps (\d+)", out)}
    for kind in ("spread40", "spread64", "spread128", "spread600", "fifth"):
        assert cost[kind] <= 1.15, out
    assert cost["uniform"] <= 0.1 and cost["drift"] <= 0.75, out
