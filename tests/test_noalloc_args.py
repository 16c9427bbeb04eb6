"""Arguments that t2i_gather_noalloc refuses before it looks at the device (CPU
only: no address here is ever read)."""
import ctypes as C

import pytest

from paper_2607_26566_gb300 import _lib as L

P = 65536


def refused(lib, why, pool=1 << 40, pool_bytes=16 * P, page=0, dst=1 << 41):
    pages = (C.c_uint32 * 1)(page)
    st = lib.t2i_gather_noalloc(pool, pool_bytes, P, pages, 1, P, dst, P, 0, 0, None)
    return st == L.ERR_INVALID and why in lib.t2i_last_error(None)


@pytest.mark.parametrize("off", [1, 2, 4, 8, 12, 24, 255])
def test_a_pool_that_is_not_16_byte_aligned(lib, off):
    """The kernels read pages as 16-byte vectors."""
    assert refused(lib, b"16-byte aligned", pool=(1 << 40) + off)


@pytest.mark.parametrize("pool_bytes,page", [((1 << 64) - P, 16), ((1 << 64) - (1 << 40), 1 << 20), ((1 << 64) - (1 << 30), 0)])
def test_a_pool_that_wraps_around_the_address_space(lib, pool_bytes, page):
    """Its end lies below its start, so it would pass as part of its allocation."""
    assert refused(lib, b"wraps", pool_bytes=pool_bytes, page=page)
