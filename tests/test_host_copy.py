"""The host's side of results that are copied back, as far as it runs without a GPU."""
import ctypes as C

import numpy as np
import pytest

import __graft_entry__ as entry
import paper_2110_02987_b200 as pkg


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("nbytes", [0, 4095, 1 << 20, (1 << 20) + 4097, 5 << 20])
@pytest.mark.parametrize("shift", [0, 1, 4095])
def test_a_destination_keeps_its_contents_until_the_copy(nbytes, shift):
    """gad_forward touches the pages of its destination while the GPU computes; if the pass then fails, the caller's array is what
    it was, to the last byte."""
    touch = pkg.load()._ZN3gad13host_prefaultEPvm    # gad::host_prefault(void*, size_t)
    touch.argtypes, touch.restype = [C.c_void_p, C.c_size_t], None
    buf = np.random.default_rng(nbytes + shift).integers(0, 256, nbytes + 4096, dtype=np.uint8)
    want = buf.copy()
    touch(buf.ctypes.data + shift, nbytes - shift if nbytes > shift else nbytes)
    assert np.array_equal(buf, want)


def test_host_loops_share_one_team():
    """Threads come up with the first host loop and stay: a loop of fewer threads would take the others down, and the next one of all would
    pay for setting them up again.  (A process of its own with three threads, which no loop would choose by itself.)"""
    import os, subprocess, sys
    code = r"""
import ctypes as C, os, sys
sys.path[:0] = [%r, %r]
import numpy as np
import paper_2110_02987_b200 as pkg
from paper_2110_02987_b200 import binding as b
n = 70000
rowptr = np.arange(n + 1, dtype=np.int64); col = np.arange(n, dtype=np.int32)
z, none = np.zeros(2, np.int64), np.empty(0, np.int32)
cp = np.array([0, n], np.int64)
threads = lambda: set(os.listdir("/proc/self/task"))
L = pkg.load()
def store(): pkg.gad_workspace_bytes(n, rowptr, col, cp, col, z, none, (4, 2))
def augment():
    csr = b.gad_csr(n, n, b._ptr(rowptr, C.c_int64), b._ptr(col, C.c_int32), None)
    out = C.c_size_t(0)
    assert L.gad_augment_workspace_bytes(C.byref(csr), 1, b._ptr(cp, C.c_int64), b._ptr(col, C.c_int32), C.byref(b._AugmentConfig(2, 4, 0.01, 0.05, 1.96, 0)), C.byref(out)) == 0
def touch():
    buf = np.zeros(3 << 20, np.uint8)
    L._ZN3gad13host_prefaultEPvm(C.c_void_p(buf.ctypes.data), C.c_size_t(buf.size))
touch()                   # (looks for the CUDA driver, once)
store()
first = threads()
for f in (augment, store, touch, store, touch, augment):
    f()
    assert threads() == first, (f.__name__, first, threads())
""" % (os.path.dirname(os.path.dirname(os.path.abspath(__file__))), os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, OMP_NUM_THREADS="3"), capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("resident", [0, 1])
def test_augment_checks_the_graph_whether_or_not_it_is_on_the_device(resident):
    from paper_2110_02987_b200 import binding as b
    L = pkg.load()
    n = 50
    rowptr, col = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32)
    cp = np.array([0, n], np.int64)
    nodes = np.arange(n, dtype=np.int32)

    def ws():
        csr = b.gad_csr(n, n, b._ptr(rowptr, C.c_int64), b._ptr(col, C.c_int32), None)
        out = C.c_size_t(0)
        cfg = b._AugmentConfig(2, 4, 0.01, 0.05, 1.96, 0, resident)
        return L.gad_augment_workspace_bytes(C.byref(csr), C.c_int32(1), b._ptr(cp, C.c_int64), b._ptr(nodes, C.c_int32), C.byref(cfg), C.byref(out))

    assert ws() == 0
    col[7] = n
    assert ws() == -2
    col[7] = 7
    rowptr[9] = 12
    assert ws() == -3
