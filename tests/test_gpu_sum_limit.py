"""Sums whose threads add more terms than their integer holds between two
folds, all at the top of the window that their first value opened.

Tolerance, as in the other sum tests: 2 eps sum|x| of the exactly rounded sum."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.mark.parametrize("first,rest", [(0.99, 1.9999), (-65535.0, -131071.0), (16384.0, 131065.4464)])
@pytest.mark.parametrize("blocks", [1, 3])
def test_full_windows(gf_lib, first, rest, blocks):
    import torch
    gf = gf_lib
    n = 1 << 20 if blocks == 1 else 1 << 21
    x = np.full(n, rest)
    x[0] = first
    xd = torch.from_numpy(x).cuda()
    out = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    rc = gf.gf_reduce_f64_noalloc(xd.data_ptr(), n, gf.GF_REDUCE_SUM, out.data_ptr(), blocks,
                                  torch.cuda.current_stream().cuda_stream)
    assert rc == gf.GF_OK
    assert abs(out.item() - math.fsum(x)) <= 2 * EPS * math.fsum(np.abs(x))
