"""Store.free lets other Python threads run while it waits for the store (CPU
only: the CPython entry points over a stub of the library)."""
import ctypes
import importlib.util
import os
import subprocess
import sysconfig
import threading

import numpy as np
import pytest

from paper_2607_26566_gb300 import build as b
from paper_2607_26566_gb300.store import Store

# t2i_free waits, as it would for the store's lock, until another thread has
# let it go on (status 0) or two seconds have passed (status 5).
STUB = r"""
#include <time.h>
#include "t2istore.h"
static volatile int entered, released;
int stub_entered(void) { return entered; }
void stub_release(void) { released = 1; }
t2i_status t2i_free(t2i_store* s, const t2i_id* ids, uint32_t n) {
    struct timespec ms = {0, 1000000};
    entered = 1;
    for (int i = 0; i < 2000 && !released; ++i) nanosleep(&ms, 0);
    return released ? T2I_OK : T2I_ERR_CUDA;
}
t2i_status t2i_put_batch(t2i_store* s, const t2i_put_desc* d, uint32_t n, t2i_id* ids, void* st) { return T2I_OK; }
t2i_status t2i_get_batch(t2i_store* s, const t2i_get_desc* d, uint32_t n, t2i_status* p, void* st) { return T2I_OK; }
"""


def test_free_releases_the_interpreter_lock(tmp_path):
    inc = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(inc, "Python.h")):
        pytest.skip("no Python.h")
    (tmp_path / "stub.c").write_text(STUB)
    so = str(tmp_path / "_pycall.so")
    subprocess.run([os.environ.get("CC", "gcc"), "-shared", "-fPIC", "-I" + b.INCLUDE, "-I" + inc, str(tmp_path / "stub.c"),
                    os.path.join(b.CSRC, b.PYCALL_SRC), "-o", so], check=True)
    spec = importlib.util.spec_from_file_location("_pycall", so)
    fast = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(fast)
    stub = ctypes.CDLL(so)
    done = threading.Event()

    def other():
        while not stub.stub_entered() and not done.is_set():
            pass
        stub.stub_release()

    st = Store.__new__(Store)
    st._fast, st._hi = fast, 1
    t = threading.Thread(target=other)
    t.start()
    status = st.free(np.array([1, 2], np.uint64))
    done.set()
    t.join()
    assert status == 0, "no other thread ran while the call waited"
