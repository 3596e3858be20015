"""A launch's host side with a fake CUDA runtime (no GPU): what the reset
kernel writes lies inside the instance's allocations, and an instance goes to
the next program only when that kernel has run, also where a launch fails, and
a program's state counts the workers that its regions have, and a program with
two kernels gets the ones that it asks for."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2306_11686_gb300", "csrc")


@pytest.fixture(scope="module")
def launch_bin(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("launch") / "launch_fake_cuda")
    subprocess.run(["nvcc", "-std=c++17", "-O1", "-diag-suppress", "177,174", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "launch_fake_cuda.cu"), os.path.join(CSRC, "host", "server.cpp"),
                    "-o", out, "-lpthread"], check=True, capture_output=True)
    return out


@pytest.mark.parametrize("scenario", ["reset", "failed", "split", "clear", "second"])
def test_launch_scenario(launch_bin, scenario):
    p = subprocess.run([launch_bin, scenario], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout + p.stderr
