"""The paired tensor-core transforms at the edges of their tiles: rows that leave the second CTA of a pair empty, one row, full or
ragged; reductions one value around a ring stage, columns around a tile, B resident or streamed, two or four lo tiles; replicas
with parameters of their own; the ReLU mask, dropout and bfloat16 drains."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import small_random_case, rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


# flag bit 7: small layers on the tensor cores too, else most of these run on the FP32 ALUs in their small tiles
@pytest.mark.parametrize("bit7", [0, 128])
@pytest.mark.parametrize("rows", [1, 127, 128, 129, 256, 257])
@pytest.mark.parametrize("dims,kw", [
    ((31, 17, 5), {}), ((33, 130, 16, 3), {}), ((700, 33, 2), {}), ((129, 256, 257, 4), dict(flags=4)),
    ((300, 300, 64, 9), dict(flags=4, dropout=0.3)), ((24, 160, 290, 5), dict(flags=4)), ((150, 96, 70), dict(dropout=0.2)), ((64, 512, 40), dict(gemm_mode=1)), ((1433, 64, 40, 7), dict(gemm_mode=1, flags=4))])
def test_row_and_column_edges(rows, dims, kw, bit7):
    kw = dict(kw, flags=kw.get("flags", 0) | bit7)
    K = 3
    case = small_random_case(rows, n=rows * K + 3, K=K, p=min(0.3, 4.0 / (rows * K)), halo=False)
    tol = 5e-2 if kw.get("gemm_mode") else TOL
    g, ref, _ = make_pair(case, dims, rows, lr=1e-3, **kw)   # (a longer step saturates the loss of a single row)
    with g:
        rng = np.random.default_rng(1)
        if not kw.get("gemm_mode"):   # every replica its own parameters, before the first consensus makes them equal
            for k in range(K):
                theta = (ref.get_params(k) + 0.05 * rng.standard_normal(g.P)).astype(np.float32)
                g.set_params(k, theta)
                ref.set_params(k, theta)
        for _ in range(2):
            lg = g.train_epoch()
            lr, _ = oracle_step(g, ref, tol)
            assert np.max(np.abs(lg - lr)) <= (1e-4 if tol == TOL else 5e-2)
        for l in range(1, len(dims)):
            assert rel_err(g.get_activation(l), ref.activation(l)) <= tol
        for k in range(K):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= tol
            assert rel_err(g.get_params(k), ref.get_params(k)) <= tol


# Tiles of 96 columns (75 - 96, 150 - 192 and so on), which need row tiles enough not to be spread: 38 pairs for one column tile, 19 for two.  Of large launches
# (four turns of the CTA pairs in tiles of 256 columns, as nearly full as the choice needs) the same three forms of a forward transform: wide tiles,
# narrow ones with B streamed, narrow ones with B resident; in the epilogue, with dropout and (flag bit 5: transform first) without, where the mask is left as bits.
# (A quarter is the same threshold of the 24-bit hash in fp32 and in the oracle; 0.3 is not, and one unit in 2^24 then differs.)
@pytest.mark.parametrize("rows,dims,kw", [
    (9800, (33, 150, 90, 5), {}), (9800, (33, 150, 90, 5), dict(dropout=0.25)), (9800, (8, 130, 150, 190), dict(flags=36)),
    (75000, (24, 150, 5), {}), (75000, (100, 160, 5), {}), (75000, (128, 132, 5), {}), (75000, (100, 160, 5), dict(dropout=0.25)),
    (75000, (8, 40, 150, 5), dict(flags=36)), (75000, (8, 100, 160, 5), dict(flags=36)), (75000, (8, 128, 132, 5), dict(flags=36)),
    (37500, (64, 260, 5), {}), (37500, (100, 300, 5), {}), (37500, (36, 400, 5), {}), (37500, (36, 400, 5), dict(dropout=0.25))])
def test_tiles_of_many_rows(rows, dims, kw):
    u = np.arange(rows)
    col = np.sort(np.stack([(u - 1) % rows, (u + 1) % rows], 1), axis=1).astype(np.int32).ravel()
    core = [np.arange(0, rows // 3 + 50, dtype=np.int32), np.arange(rows // 3 + 50, rows, dtype=np.int32)]
    g, ref, _ = make_pair((rows, np.arange(0, 2 * rows + 1, 2, dtype=np.int64), col, None, core, [np.zeros(0, np.int32)] * 2), dims, rows, lr=1e-2, **kw)
    with g:
        lg = g.train_epoch()
        lr, _ = oracle_step(g, ref, TOL)
        assert np.max(np.abs(lg - lr)) <= 1e-4
        for l in range(1, len(dims)):
            assert rel_err(g.get_activation(l), ref.activation(l)) <= TOL
        for k in range(2):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL
