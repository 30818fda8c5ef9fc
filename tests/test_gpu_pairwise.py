"""Pairwise importance weights on the tensor cores at the edges of their tiles (256 x 256 pairs, taken whole or in two column parts):
subgraphs one row around a half and a whole tile, an empty one between them, enough tiles for whole ones, features around the MMA's K,
distances below and far above beta, and groups of nearly equal rows, whose pairs come from the differences."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import small_random_case
from test_gpu_parity import make_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("F,beta,alike", [(8, 1.0, False), (33, 1e-5, True), (70, 1.0, True)])
@pytest.mark.parametrize("sizes", [(1, 127), (128, 129), (255, 0, 256), (257, 384), (513,), (2700, 300)])
def test_tile_edges(sizes, F, beta, alike):
    n = sum(sizes)
    n, rowptr, col, w, _, _ = small_random_case(F, n=n, K=1, p=min(0.3, 6.0 / n), halo=False)
    ends = np.cumsum(sizes)
    core = [np.arange(e - m, e, dtype=np.int32) for e, m in zip(ends, sizes)]
    X = np.random.default_rng(F).standard_normal((n, F)).astype(np.float32)
    if alike:
        X[1::7] = X[0] + 1e-2 * X[1::7]
    g, ref, _ = make_pair((n, rowptr, col, w, core, [np.zeros(0, np.int32)] * len(core)), (F, 5, 3), F, X=X, zeta_mode=1, beta=beta)
    with g:
        for _ in range(2):
            zg, wg = g.subgraph_weights()
            zr, wr = ref.subgraph_weights()
            assert np.max(np.abs(zg - zr)) <= 2e-6 * max(np.max(zr), 1e-30)
            assert np.max(np.abs(wg - wr)) <= 2e-6
