"""The Jacobi program on grids with regions of zeros (a source in a zero
field, the usual start of a Laplace solve): bit for bit the serial program,
and its sweeps stay fixed-point sweeps, which the number of regions shows (two
that sample the grid once, one a sweep, and one more a sweep at most for
points left out)."""
import subprocess

import numpy as np
import pytest

from paper_2306_11686_gb300 import inputs

pytestmark = pytest.mark.gpu


def grid(n, kind):
    g = np.zeros(n ** 3)
    c = g.reshape(n, n, n)
    u = inputs.jacobi_input(n, seed=11).reshape(n, n, n)
    if kind == "hot":                          # a hot block in zeros
        c[n // 2 - 8:n // 2 + 8, n // 2 - 8:n // 2 + 8, n // 2 - 8:n // 2 + 8] = 1.0
    elif kind == "half":
        c[n // 2:] = 0.25 + 0.75 * u[n // 2:]
    elif kind == "point":
        c[n // 3, n // 2, n // 2] = 1.0
    elif kind == "large point":
        c[n // 3, n // 2, n // 2] = 1e30
    elif kind == "minus zero":
        c[...] = -0.0
        c[2, 2, 2] = 1.0
    elif kind == "minus point":
        c[n // 3, n // 2, n // 2] = -1.0
    return g


KINDS = ["hot", "half", "zero", "point", "large point", "minus zero", "minus point"]


@pytest.mark.parametrize("n,sweeps", [(103, 4), (160, 3)])
@pytest.mark.parametrize("kind", KINDS)
def test_jacobi_with_zeros(gf_lib, oracle_bin, tmp_path, n, sweeps, kind):
    import torch
    gf = gf_lib
    g = grid(n, kind)
    inputs.write_f64(tmp_path / "in.bin", g)
    p = subprocess.run([oracle_bin("jacobi"), str(n), str(sweeps), str(tmp_path / "in.bin"), str(tmp_path / "ref.bin")],
                       capture_output=True, text=True, check=True)
    with gf.Context(timeout_ns=10_000_000_000, stdout_path=tmp_path / "out.txt", heap_bytes=4 * n ** 3 * 8 + (64 << 20),
                    heap_small_pct=5) as ctx:
        rc, ec = ctx.run("jacobi", [n, sweeps, tmp_path / "gpu.bin"], [(torch.from_numpy(g).cuda(), gf.GF_BUF_IN)])
        st = ctx.stats()
    assert ec == 0
    assert sorted(open(tmp_path / "out.txt").read().splitlines()) == sorted(p.stdout.splitlines())
    assert (tmp_path / "gpu.bin").read_bytes() == (tmp_path / "ref.bin").read_bytes()
    if not kind.startswith("minus"):               # the final write copies in regions of its own
        assert st.regions - st.copy_regions <= 2 * sweeps + 2
