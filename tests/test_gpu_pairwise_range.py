"""Pairwise importance weights at the ends of what fp32 holds: beta far from one, rows of zeros (whose distance is zero, so that beta is
all there is in the denominator), large features."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import small_random_case
from test_gpu_parity import make_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("beta", [1e-30, 1e-25, 1e-18, 1.0, 1e18, 1e25])
@pytest.mark.parametrize("scale,zeros", [(1.0, True), (1.0, False), (1.5e18, True), (1e-15, False)])
@pytest.mark.parametrize("sizes", [(300, 200), (700,)])
def test_denominators_whose_products_leave_the_range(sizes, scale, zeros, beta):
    n = sum(sizes)
    n, rowptr, col, w, _, _ = small_random_case(3, n=n, K=1, p=6.0 / n, halo=False)
    ends = np.cumsum(sizes)
    core = [np.arange(e - m, e, dtype=np.int32) for e, m in zip(ends, sizes)]
    X = (scale * np.random.default_rng(3).standard_normal((n, 8))).astype(np.float32)
    if zeros:
        X[n // 5:n // 2] = 0.0
    g, ref, _ = make_pair((n, rowptr, col, w, core, [np.zeros(0, np.int32)] * len(core)), (8, 5, 3), 3, X=X, zeta_mode=1, beta=beta)
    with g:
        zg, wg = g.subgraph_weights()
        zr, wr = ref.subgraph_weights()
        assert np.max(np.abs(zg - zr)) <= 2e-6 * np.max(zr), (zg, zr)
        assert np.max(np.abs(wg - wr)) <= 2e-6


@pytest.mark.parametrize("F", [1, 15, 16, 17, 63, 64, 65, 130])
@pytest.mark.parametrize("rows", ["alike", "apart", "within", "tiny"])
def test_rows_and_values_of_every_size(F, rows):
    """The fp16 copies are scaled row by row: rows whose sizes differ by up to 2^40, values that do inside a row, and rows of subnormal values; each row
    keeps 22 bits of its largest values, so the distances' relative error stays that of fp32 sums."""
    n = 390
    n, rowptr, col, w, _, _ = small_random_case(7, n=n, K=1, p=6.0 / n, halo=False)
    rng = np.random.default_rng(F)
    X = rng.standard_normal((n, F))
    if rows == "apart":
        X *= 2.0 ** rng.integers(-20, 21, (n, 1))
    if rows == "within":
        X *= 2.0 ** rng.integers(-20, 21, (n, F))
    if rows == "tiny":
        X[::3] *= 1e-41
    g, ref, _ = make_pair((n, rowptr, col, w, [np.arange(n, dtype=np.int32)], [np.zeros(0, np.int32)]), (F, 5, 3), 3, X=X.astype(np.float32), zeta_mode=1)
    with g:
        zg, _ = g.subgraph_weights()
        zr, _ = ref.subgraph_weights()
        assert np.max(np.abs(zg - zr)) <= 2e-6 * np.max(zr), (zg, zr)
