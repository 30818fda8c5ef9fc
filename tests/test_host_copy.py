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
