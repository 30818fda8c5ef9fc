"""The ReLU mask that a forward transform leaves as bits for the transform back through its layer: hidden widths around a word, around a ring stage and
around the tiles, rows cut into parts in front of it, dropout, operands in one pass, and layers on the FP32 ALUs, which leave none."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


def hub_case(n, K):
    rng = np.random.default_rng(n)
    src = np.concatenate([rng.integers(0, n, 3 * n), np.repeat(np.arange(K) * (n // K), n // 2)])   # a hub in every block
    dst = rng.integers(0, n, src.size)
    keep = src != dst
    key = np.unique(np.concatenate([src[keep] * n + dst[keep], dst[keep] * n + src[keep]]))
    rowptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    core = [c.astype(np.int32) for c in np.array_split(np.arange(n), K)]
    return n, rowptr, (key % n).astype(np.int32), None, core, [np.zeros(0, np.int32)] * K


# first layer: transforms first where it is wider than twice the hidden one, else aggregates first (flag bit 7: all on the tensor cores)
@pytest.mark.parametrize("hidden", [3, 16, 17, 31, 32, 33, 63, 64, 65, 127, 129, 257, 1030])
@pytest.mark.parametrize("first,kw", [(2, {}), (0.5, {}), (2.5, dict(dropout=0.4)), (0.5, dict(dropout=0.4)), (2.5, dict(gemm_mode=1)), (0.5, dict(gemm_mode=1)),
                                      (0.5, dict(flags=4))])
def test_gradients_behind_the_mask(hidden, first, kw):
    if hidden == 1030 and first > 2:
        first = 0.1
    kw = dict(kw)
    kw["flags"] = kw.get("flags", 4) | (0 if kw == dict(flags=4) else 128)   # 4: no fused kernel in place of the masked transform
    dims = (max(2, int(first * hidden) + (1 if first > 2 else 0)), hidden, hidden, 20)
    g, ref, _ = make_pair(hub_case(430, 3), dims, hidden, lr=1e-2, **kw)
    tol = 5e-2 if kw.get("gemm_mode") else TOL
    with g:
        for _ in range(2):
            lg = g.train_epoch()
            lr, _ = oracle_step(g, ref, tol)
            assert np.max(np.abs(lg - lr)) <= (1e-4 if tol == TOL else 5e-2)
        for k in range(3):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= tol
