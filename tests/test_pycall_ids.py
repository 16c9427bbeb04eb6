"""The CPython entry points that take a uint64 array (get_batch_for, free_ids):
which objects they take, and which they leave to the general path (None).
CPU only: a null store comes back INVALID from the library."""
import array

import numpy as np
import pytest

from paper_2607_26566_gb300 import _lib as L
from paper_2607_26566_gb300.store import GET_DTYPE, Store


@pytest.fixture()
def fast(lib):
    f = L.pycall()
    if f is None:
        pytest.skip("built without Python.h: the ctypes binding serves every call")
    return f


IDS = np.array([7, 9, 11, 13, 15, 17], np.uint64)


@pytest.mark.parametrize("ids,taken", [
    (IDS[:3].copy(), True), (IDS, True), (IDS[1:], True), (IDS.reshape(3, 2), True),
    (IDS[:2].copy(), False), (IDS[::2], False), (IDS.astype(np.int64), False), (IDS.astype(">u8"), False),
    (IDS.astype(np.float64), False), ([7, 9, 11], False), (np.uint64(7), False), (None, False)])
def test_get_batch_for(fast, ids, taken):
    d = np.zeros(3, GET_DTYPE)
    st = fast.get_batch_for(0, d.ctypes.data, 3, ids, 0, 0)
    assert st == (L.ERR_INVALID if taken else None)
    assert list(d["id"]) == ([int(x) for x in ids.reshape(-1)[:3]] if taken else [0, 0, 0])


@pytest.mark.parametrize("ids,taken", [(IDS, True), (IDS[:0], True), (IDS[::2], False), (IDS.reshape(3, 2), False),
                                       (IDS.astype(np.uint32), False), ([7], False), (np.array(7, np.uint64), False)])
def test_free_ids(fast, ids, taken):
    assert fast.free_ids(0, ids) == (L.ERR_INVALID if taken else None)


def bare_store(fast):
    """A store without a device (its handle is null), and a prepared get of 3."""
    st = Store.__new__(Store)
    st._lib, st._fast, st._h, st._hi = L.load(), fast, None, 0
    return st, st.prepare_get(np.zeros(3, GET_DTYPE))


UNALIGNED = np.frombuffer(bytearray(1 + 6 * 8), np.uint8)[1:].view(np.uint64)
UNALIGNED[:] = IDS


@pytest.mark.parametrize("ids", [IDS[:3].copy(), IDS, IDS.reshape(3, 2), UNALIGNED, UNALIGNED[:3], [7, 9, 11],
                                 array.array("Q", [7, 9, 11])])
def test_get_prepared_takes(fast, ids):
    """An array of at least n ids, or any n numbers."""
    st, p = bare_store(fast)
    assert st.get_prepared(p, ids, stream=0) == L.ERR_INVALID  # from the library: a null store
    assert list(p.descs["id"]) == [7, 9, 11]


@pytest.mark.parametrize("ids", [IDS[:2].copy(), IDS[::2][:2], list(range(6)), array.array("Q", range(6)),
                                 memoryview(IDS), np.zeros((3, 0), np.uint64), np.array(7, np.uint64)])
def test_get_prepared_refuses(fast, ids):
    """Fewer than n ids, or more than n in anything but an array of them."""
    st, p = bare_store(fast)
    with pytest.raises((ValueError, TypeError)):
        st.get_prepared(p, ids, stream=0)
    assert not p.descs["id"].any()
