"""The Jacobi program's fixed-point sweeps under the kernel split: the region
kernel's own grid, bit for bit the serial program."""
import subprocess

import pytest

from paper_2306_11686_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sweeps,grid", [(103, 4, 0), (128, 2, 0), (103, 2, 1), (103, 2, 7)])
def test_split_fixed_point_sweeps(gf_lib, oracle_bin, tmp_path, n, sweeps, grid):
    import torch
    gf = gf_lib
    g = inputs.jacobi_input(n, seed=9)
    inputs.write_f64(tmp_path / "in.bin", g)
    p = subprocess.run([oracle_bin("jacobi"), str(n), str(sweeps), str(tmp_path / "in.bin"), str(tmp_path / "ref.bin")],
                       capture_output=True, text=True, check=True)
    with gf.Context(split_regions=1, grid=grid, timeout_ns=10_000_000_000, heap_bytes=4 * n ** 3 * 8 + (64 << 20),
                    heap_small_pct=5, stdout_path=tmp_path / "out.txt") as ctx:
        rc, ec = ctx.run("jacobi", [n, sweeps, tmp_path / "gpu.bin"], [(torch.from_numpy(g).cuda(), gf.GF_BUF_IN)])
    assert ec == 0
    assert sorted(open(tmp_path / "out.txt").read().splitlines()) == sorted(p.stdout.splitlines())
    assert (tmp_path / "gpu.bin").read_bytes() == (tmp_path / "ref.bin").read_bytes()
