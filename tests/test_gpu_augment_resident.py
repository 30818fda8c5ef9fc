"""gad_augment on a graph that an earlier call left on the device: the caller's arrays are still checked, and arrays that are not
those of the earlier call are refused, with every access inside the workspace."""
import numpy as np
import pytest

import __graft_entry__ as entry
import paper_2110_02987_b200 as pkg
from conftest import small_random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("n", [80, 70000])     # the checks on one thread and on several
def test_the_callers_arrays_are_checked_on_every_call(n):
    if n == 80:
        _, rowptr, col, _, cores, _ = small_random_case(3, n=n, K=3)
    else:
        u = np.arange(n)
        col = np.stack([(u - 1) % n, (u + 1) % n], 1).astype(np.int32).ravel()
        rowptr = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
        cores = [np.arange(0, n // 2, dtype=np.int32), np.arange(n // 2, n, dtype=np.int32)]
    aug = pkg.Augmenter(n, rowptr, col)
    want, walks = aug.run(cores, 2, alpha=0.3, seed=9)
    last = len(aug.col) - 1
    for at, value in ((0, n), (last, -1), (last, 2**31 - 1)):
        keep = aug.col[at]
        aug.col[at] = value
        with pytest.raises(pkg.GadError) as e:
            aug._resident = True
            aug.run(cores, 2, alpha=0.3, seed=9)
        assert e.value.code == -2
        aug.col[at] = keep
    keep = aug.rowptr[n // 2]
    aug.rowptr[n // 2] = aug.rowptr[n // 2 + 1] + 1
    with pytest.raises(pkg.GadError) as e:
        aug._resident = True
        aug.run(cores, 2, alpha=0.3, seed=9)
    assert e.value.code == -3
    aug.rowptr[n // 2] = keep
    for resident in (True, False):
        aug._resident = resident
        got, w = aug.run(cores, 2, alpha=0.3, seed=9)
        assert np.array_equal(walks, w) and all(np.array_equal(a, b) for a, b in zip(want, got))


def test_another_graph_of_the_same_size_is_refused():
    """The walks on the device follow its graph, the room for them the caller's: a graph whose core sets have fewer entries leaves too
    little.  The kernels stop where the room ends and the call says so."""
    n = 4000
    rng = np.random.default_rng(1)
    half = n // 2
    # nearly all entries in the rows of the first half; then in those of the second
    deg = np.concatenate([np.full(half, 9), np.full(n - half, 1)])
    def graph(d):
        rowptr = np.zeros(n + 1, np.int64)
        np.cumsum(d, out=rowptr[1:])
        col = rng.integers(0, n, rowptr[-1]).astype(np.int32)
        return rowptr, col
    dense, sparse = graph(deg), graph(deg[::-1])
    cores = [np.arange(0, half, dtype=np.int32)]
    aug = pkg.Augmenter(n, dense[0].copy(), dense[1].copy())
    want, walks = aug.run(cores, 2, alpha=0.1, seed=3)
    aug.rowptr[:], aug.col[:] = sparse
    with pytest.raises(pkg.GadError) as e:
        aug._resident = True
        aug.run(cores, 2, alpha=0.1, seed=3)
    assert e.value.code == -1
    aug.rowptr[:], aug.col[:] = dense
    got, w = aug.run(cores, 2, alpha=0.1, seed=3)
    assert np.array_equal(walks, w) and np.array_equal(want[0], got[0])
