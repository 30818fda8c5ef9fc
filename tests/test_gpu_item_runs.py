"""Work lists of subgraphs around and beyond the number of rows whose items are ordered by length together: cut rows, rows of every length
and a second subgraph that starts inside a run."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("first", [16383, 16384, 16385, 40001])
@pytest.mark.parametrize("dims", [(6, 9, 3), (70, 40, 5)])
def test_runs_of_rows(first, dims):
    n = first + 517
    rng = np.random.default_rng(first)
    src = np.concatenate([rng.integers(0, n, 4 * n), np.repeat(rng.integers(0, n, 6), 700)])   # six rows of many entries
    dst = rng.integers(0, n, src.size)
    keep = src != dst
    key = np.unique(np.concatenate([src[keep] * n + dst[keep], dst[keep] * n + src[keep]]))
    rowptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    core = [np.arange(first, dtype=np.int32), np.arange(first, n, dtype=np.int32)]
    halo = [np.array([n - 1], np.int32), np.array([0, 5], np.int32)]
    g, ref, _ = make_pair((n, rowptr, (key % n).astype(np.int32), None, core, halo), dims, first, lr=0.1)
    with g:
        assert g.check_store() == 0
        lg = g.train_epoch()
        lr, _ = oracle_step(g, ref, TOL)
        assert np.max(np.abs(lg - lr)) <= 1e-4
        for l in range(1, len(dims)):
            assert rel_err(g.get_activation(l), ref.activation(l)) <= TOL
        for k in range(2):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL
