"""Layers on the FP32 ALUs over many rows: their weight gradient in more chunks than there are SMs, whole and ragged, in one subgraph
and in many, beside layers on the tensor cores."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("n,K", [(9472, 1), (9473, 2), (20011, 3), (12000, 41)])
@pytest.mark.parametrize("dims", [(20, 9, 5), (8, 33, 3), (70, 31, 6)])   # the first layer of the last one: tensor cores from 14 300 rows on
def test_weight_gradients_of_many_chunks(n, K, dims):
    u = np.arange(n)
    hop = np.stack([(u - 7) % n, (u - 1) % n, (u + 1) % n, (u + 7) % n], 1)
    col = np.sort(hop, axis=1).astype(np.int32).ravel()
    rowptr = np.arange(0, 4 * n + 1, 4, dtype=np.int64)
    ends = np.linspace(0, n, K + 1).astype(int)
    core = [np.arange(a, b, dtype=np.int32) for a, b in zip(ends[:-1], ends[1:])]
    halo = [np.array([b % n], np.int32) if K > 1 else np.zeros(0, np.int32) for b in ends[1:]]
    g, ref, _ = make_pair((n, rowptr, col, None, core, halo), dims, n + K, lr=0.1)
    with g:
        for _ in range(2):
            lg = g.train_epoch()
            lr, _ = oracle_step(g, ref, TOL)
            assert np.max(np.abs(lg - lr)) <= 1e-4
        for k in sorted({0, K // 2, K - 1}):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL
            assert rel_err(g.get_params(k), ref.get_params(k)) <= TOL
