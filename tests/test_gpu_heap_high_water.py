"""The high-water mark of the small heap is what was live at most: no more than
the heap holds where many requests fail together, and just that where all of
it was handed out."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slabs,bytes_", [(1, 65536), (7, 16384), (29, 8192), (64, 256), (29, 65536)])
def test_failed_requests_do_not_show(gf_lib, slabs, bytes_):
    import torch
    gf = gf_lib
    blocks = slabs * (256 << 10) // bytes_
    per, T = 2, 4 * blocks                        # eight times as many requests as blocks, at the same time
    ptrs = torch.zeros(2 * T * per, dtype=torch.int64, device="cuda")
    with gf.Context(timeout_ns=10_000_000_000, heap_bytes=slabs * (256 << 10), heap_small_pct=100) as c:
        rc, ec = c.run("heap_exhaust", [T, per, bytes_], [(ptrs, 1)])
        st = c.stats()
    assert ec == 0
    assert st.heap_high_water == blocks * bytes_
    assert st.heap_alloc == 2 * blocks and st.heap_free == 2 * blocks and st.heap_fail == 2 * (T * per - blocks)
    assert st.heap_live_bytes == 0
