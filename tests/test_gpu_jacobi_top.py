"""The Jacobi program on grids whose sums of six come close to the largest
double or overflow, against the serial program bit for bit."""
import subprocess

import numpy as np
import pytest

from paper_2306_11686_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [1019, 1020, 1021, 1022])
@pytest.mark.parametrize("spread", [0.0, 0.1])
def test_jacobi_near_overflow(gf_lib, oracle_bin, tmp_path, exponent, spread):
    import torch
    gf = gf_lib
    n, sweeps = 103, 3
    g = inputs.jacobi_input(n, seed=11)
    c = g.reshape(n, n, n)
    inner = (slice(1, -1),) * 3
    c[inner] = (1.9 - spread * c[inner]) * 2.0 ** exponent
    inputs.write_f64(tmp_path / "in.bin", g)
    p = subprocess.run([oracle_bin("jacobi"), str(n), str(sweeps), str(tmp_path / "in.bin"), str(tmp_path / "ref.bin")],
                       capture_output=True, text=True, check=True)
    with gf.Context(timeout_ns=10_000_000_000, stdout_path=tmp_path / "out.txt", heap_bytes=4 * n ** 3 * 8 + (64 << 20),
                    heap_small_pct=5) as ctx:
        rc, ec = ctx.run("jacobi", [n, sweeps, tmp_path / "gpu.bin"], [(torch.from_numpy(g).cuda(), gf.GF_BUF_IN)])
    assert ec == 0
    assert sorted(open(tmp_path / "out.txt").read().splitlines()) == sorted(p.stdout.splitlines())
    assert (tmp_path / "gpu.bin").read_bytes() == (tmp_path / "ref.bin").read_bytes()
