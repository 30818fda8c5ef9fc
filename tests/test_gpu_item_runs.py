"""Work lists of subgraphs around and beyond the number of rows whose items are ordered by length together where runs are used: cut rows, rows of every
length and a second subgraph that starts inside a run; launches that take the list in runs (wide operands) and ones that do not."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


def graph(first, directed):
    n = first + 517
    rng = np.random.default_rng(first)
    src = np.concatenate([rng.integers(0, n, 4 * n), np.repeat(rng.integers(0, n, 6), 700)])   # six rows of many entries
    dst = rng.integers(0, n, src.size)
    keep = src != dst
    key = np.unique(np.concatenate([src[keep] * n + dst[keep], [] if directed else dst[keep] * n + src[keep]]).astype(np.int64))
    rowptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    core = [np.arange(first, dtype=np.int32), np.arange(first, n, dtype=np.int32)]
    halo = [np.array([n - 1], np.int32), np.array([0, 5], np.int32)]
    return n, rowptr, (key % n).astype(np.int32), None, core, halo


def check(g, ref, layers):
    with g:
        assert g.check_store() == 0
        lg = g.train_epoch()
        lr, _ = oracle_step(g, ref, TOL)
        assert np.max(np.abs(lg - lr)) <= 1e-4
        for l in range(1, layers + 1):
            assert rel_err(g.get_activation(l), ref.activation(l)) <= TOL
        for k in range(2):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL


@pytest.mark.parametrize("first", [16383, 16384, 16385, 40001])
@pytest.mark.parametrize("dims", [(6, 9, 3), (70, 40, 5)])
def test_runs_of_rows(first, dims):
    g, ref, _ = make_pair(graph(first, False), dims, first, lr=0.1)
    check(g, ref, len(dims) - 1)


# An operand of 1024 columns takes half of the L2 from 16 128 rows on, so these subgraphs have a list in runs from 16 385 rows on (a replicated row comes on
# top of `first`), of the store and, on the way back, of the loss rows' store or (flag bit 6) the transposed one.  Bit 5: the last layer transforms first.
@pytest.mark.parametrize("first,flags", [(16383, 32), (16384, 32), (16385, 96), (32768, 96)])
def test_wide_aggregations_in_runs_of_rows(first, flags):
    g, ref, _ = make_pair(graph(first, True), (4, 8, 1024), first, lr=0.1, flags=flags)
    check(g, ref, 2)
