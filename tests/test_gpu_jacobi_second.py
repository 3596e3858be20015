"""The Jacobi program's two kernels against the serial program, bit for bit:
grids that no fixed-point window suits, which go over to the second kernel when
a second sample shows no fewer values outside, come to suit one (values spread
at random), or stay (many zeros),
sizes that its column segments do not divide, few sweeps and many, a grid of
blocks that only the second kernel has room for, and the kernel split."""
import subprocess

import numpy as np
import pytest

from paper_2306_11686_gb300 import inputs

pytestmark = pytest.mark.gpu


def grid(n, kind):
    g = inputs.jacobi_input(n, seed=11)
    c = g.reshape(n, n, n)
    inner = (slice(1, -1),) * 3
    if kind == "signed":
        c[inner] = 2.0 * c[inner] - 1.0
    elif kind == "steep":                      # positive, 2^-58 .. 1, smooth along k
        c[inner] = (0.5 + 0.5 * c[inner]) * 2.0 ** -(0.57 * np.arange(1, n - 1)[:, None, None])
    elif kind == "some":                       # a few values outside, for good
        c[inner] = 0.5 + 0.5 * c[inner]
        c[2:-2, 2:6, 2:6] *= 2.0 ** -40
    elif kind == "wide":                       # spread over 40 binades at random
        c[inner] = (0.5 + 0.5 * c[inner]) * 2.0 ** -inputs.uniform_int(5, (n - 2) ** 3, 0, 39).reshape((n - 2,) * 3).astype(np.float64)
    elif kind == "half signed":                # many zeros
        c[inner] = 2.0 * c[inner] - 1.0
        c[n // 2:] = 0.0
    elif kind == "inf":                        # no window holds it; NaNs follow
        c[inner] = 0.25 + 0.75 * c[inner]
        c[n // 2, 5, 5] = np.inf
    return g


@pytest.mark.parametrize("n,sweeps,kind,kw", [
    (102, 3, "signed", {}), (104, 3, "signed", {}), (105, 3, "signed", {}), (103, 9, "signed", {}),
    (103, 1, "steep", {}), (103, 3, "steep", {}), (103, 4, "steep", {}), (105, 11, "steep", {}),
    (103, 9, "steep", {"grid": 1}), (103, 9, "steep", {"grid": 77}), (103, 9, "steep", {"max_programs": 3}),
    (103, 9, "steep", {"split_regions": 1}), (103, 3, "unit", {"grid": 608}), (67, 3, "unit", {"grid": 608}),
    (103, 5, "inf", {}), (103, 9, "wide", {}), (103, 9, "some", {}), (160, 9, "some", {}), (103, 5, "half signed", {}),
])
def test_two_kernels(gf_lib, oracle_bin, tmp_path, n, sweeps, kind, kw):
    import torch
    gf = gf_lib
    g = grid(n, kind)
    inputs.write_f64(tmp_path / "in.bin", g)
    p = subprocess.run([oracle_bin("jacobi"), str(n), str(sweeps), str(tmp_path / "in.bin"), str(tmp_path / "ref.bin")],
                       capture_output=True, text=True, check=True)
    with gf.Context(timeout_ns=10_000_000_000, stdout_path=tmp_path / "out.txt", heap_bytes=4 * n ** 3 * 8 + (64 << 20),
                    heap_small_pct=5, **kw) as ctx:
        for _ in range(2):                     # and again on the same instance
            rc, ec = ctx.run("jacobi", [n, sweeps, tmp_path / "gpu.bin"], [(torch.from_numpy(g).cuda(), gf.GF_BUF_IN)])
            st = ctx.stats()
            assert ec == 0
            assert (tmp_path / "gpu.bin").read_bytes() == (tmp_path / "ref.bin").read_bytes()
            assert st.heap_alloc == sweeps and st.heap_free == sweeps and st.heap_live_bytes == 0
    assert sorted(open(tmp_path / "out.txt").read().splitlines()) == sorted(2 * p.stdout.splitlines())


def test_options_take_the_second_kernel(gf_lib):
    """Its residency, four blocks an SM, is the default grid of a run with options."""
    import torch
    gf = gf_lib
    n = 67
    g = torch.from_numpy(inputs.jacobi_input(n, seed=3)).cuda()
    with gf.Context(timeout_ns=10_000_000_000, stdout_path="/dev/null", heap_bytes=64 << 20, heap_small_pct=5) as ctx:
        sms = ctx.grid_info("jacobi")[0]
        for args in ([1], [0, 4]):
            rc, ec = ctx.run("jacobi", [n, 2, "-", *args], [(g, gf.GF_BUF_IN)])
            assert ec == 0 and ctx.stats().grid == 4 * sms
