"""A grid that its sample takes for one that suits the fixed-point sweep, and
that does not: after the sweep that shows it the program leaves the sample
alone for a while (the number of regions: two samples, the sweep and the pass
over what it left out, then one region a sweep), and the results are the
serial program's, bit for bit."""
import subprocess

import numpy as np
import pytest

from paper_2306_11686_gb300 import inputs

pytestmark = pytest.mark.gpu


def sampled(cells):
    """The cells that the program's sample looks at (a hash of 0 .. 32767, scaled)."""
    h = np.arange(32768, dtype=np.uint64) * 0x9E3779B1 & 0xffffffff
    h ^= h >> 15
    h = h * 0x85EBCA6B & 0xffffffff
    h ^= h >> 13
    return (h * cells >> np.uint64(32)).astype(np.int64)


def test_sample_is_left_alone_after_a_dropped_window(gf_lib, oracle_bin, tmp_path):
    import torch
    gf = gf_lib
    n, sweeps = 160, 2                                    # segments of more planes than a sweep mends by itself
    cells = n ** 3
    g = inputs.jacobi_input(n, seed=11)
    c = g.reshape(n, n, n)
    inner = (slice(1, -1),) * 3
    c[inner] = 0.25 + 0.75 * c[inner]
    minus = np.random.default_rng(3).random(cells) < 0.05          # far more than the sweep accepts
    minus[sampled(np.uint64(cells))] = False
    g[minus] *= -1.0
    inputs.write_f64(tmp_path / "in.bin", g)
    p = subprocess.run([oracle_bin("jacobi"), str(n), str(sweeps), str(tmp_path / "in.bin"), str(tmp_path / "ref.bin")],
                       capture_output=True, text=True, check=True)
    with gf.Context(timeout_ns=10_000_000_000, stdout_path=tmp_path / "out.txt", heap_bytes=4 * cells * 8 + (64 << 20),
                    heap_small_pct=5) as ctx:
        rc, ec = ctx.run("jacobi", [n, sweeps, tmp_path / "gpu.bin"], [(torch.from_numpy(g).cuda(), gf.GF_BUF_IN)])
        st = ctx.stats()
    assert ec == 0
    assert sorted(open(tmp_path / "out.txt").read().splitlines()) == sorted(p.stdout.splitlines())
    assert (tmp_path / "gpu.bin").read_bytes() == (tmp_path / "ref.bin").read_bytes()
    assert st.regions - st.copy_regions == 2 + 1 + 1 + 1
