"""The two forms of the aggregation of 129 to 256 columns: numbers of items and average row lengths on either side of the lines between them, tails of a
batch of entries, the narrowest and widest operand, a column slab that is left over; bfloat16 operands that can and cannot be read in pairs."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


# (1157 columns: a pass of 1024 and one of 133; the form of few items up to 16 384 rows)
@pytest.mark.parametrize("n,entries,width,mode", [(301, e, w, m) for e in (1, 71, 99) for w, m in ((129, 0), (200, 0), (256, 0), (1157, 0), (130, 1), (252, 1), (256, 1))] +
                         [(16384, 3, 129, 0), (16385, 3, 129, 0), (16385, 33, 256, 0), (16385, 39, 200, 0), (16385, 71, 132, 0), (16385, 73, 132, 0)])
def test_forms(n, entries, width, mode):
    half = (entries - 1) // 2
    u = np.arange(n)
    offsets = np.concatenate([np.arange(-half, 0), np.arange(1, half + 1)])    # (the self-loop is added)
    col = np.sort((u[:, None] + offsets) % n, axis=1).astype(np.int32).ravel()
    core = [np.arange(n, dtype=np.int32)]
    dims = (width, (width + 1) // 2, 3) if n < 1000 else (width, 3)
    g, ref, _ = make_pair((n, np.arange(n + 1, dtype=np.int64) * 2 * half, col, None, core, [np.zeros(0, np.int32)]), dims, width + entries, lr=1e-2, gemm_mode=mode, flags=0 if n < 1000 else 2)
    tol = 5e-2 if mode else TOL
    with g:
        assert g.nnz_prime == n * entries and g.check_store() == 0
        lg = g.train_epoch()
        lr, _ = oracle_step(g, ref, tol)
        assert np.max(np.abs(lg - lr)) <= (5e-2 if mode else 1e-4)
        for l in range(1, len(dims)):
            assert rel_err(g.get_activation(l), ref.activation(l)) <= tol
        assert rel_err(g.get_grads(0), ref.get_grads(0)) <= tol
