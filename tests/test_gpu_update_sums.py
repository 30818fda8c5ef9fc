"""The update of small models, which adds up the chunks of the last weight gradient: numbers of replicas around what a block takes at a time, layers whose
end falls inside a block, chunks around eight to a replica, copies that differ, and models on either side of the size and of the number of chunks from which it does not."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import small_random_case, rel_err
from test_gpu_parity import make_pair, oracle_step, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


def check(g, ref, K, differ):
    with g:
        if differ:
            rng = np.random.default_rng(K)
            for k in range(K):
                theta = (ref.get_params(k) + 0.05 * rng.standard_normal(g.P)).astype(np.float32)
                g.set_params(k, theta)
                ref.set_params(k, theta)
        for _ in range(3):   # the last one replayed
            lg = g.train_epoch()
            lr, _ = oracle_step(g, ref, TOL)
            assert np.max(np.abs(lg - lr)) <= 1e-4
        for k in range(K):
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL
            assert rel_err(g.get_params(k), ref.get_params(k)) <= TOL


@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 16, 17, 33])
@pytest.mark.parametrize("dims,differ", [((3, 2), False), ((37, 5, 3), True), ((64, 33, 7, 4), False), ((300, 130, 5), False)])
def test_replicas_and_layers(K, dims, differ):
    case = small_random_case(K, n=12 * K + 30, K=K, p=0.1, halo=False)
    g, ref, _ = make_pair(case, dims, K, lr=0.05, flags=128)   # (bit 7: on the tensor cores, whose weight gradients are summed there)
    check(g, ref, K, differ)


@pytest.mark.parametrize("n,dims", [(40, (500, 511, 3)), (40, (500, 530, 3)), (6000, (9, 6, 3)), (9500, (40, 24, 3)),
                                    (3072, (40, 24, 3)), (3073, (40, 24, 3))])   # (chunks of 32 rows: 64 and 65 in the larger subgraph)
def test_sizes_and_chunks(n, dims):
    u = np.arange(n)
    col = np.sort(np.stack([(u - 1) % n, (u + 1) % n], 1), axis=1).astype(np.int32).ravel()
    core = [np.arange(0, n // 3, dtype=np.int32), np.arange(n // 3, n, dtype=np.int32)]
    g, ref, _ = make_pair((n, np.arange(0, 2 * n + 1, 2, dtype=np.int64), col, None, core, [np.zeros(0, np.int32)] * 2), dims, n, lr=0.05, flags=128)
    check(g, ref, 2, False)


@pytest.mark.parametrize("K,dims", [(2, (37, 5, 3)), (9, (64, 33, 7, 4))])
def test_gradients_of_an_epoch_that_is_not_taken(K, dims):
    """A bounded wait runs out ahead of the second epoch: its update is left out, and the gradients of all layers are still its own."""
    import paper_2110_02987_b200 as pkg
    g, ref, _ = make_pair(small_random_case(K, n=12 * K + 30, K=K, p=0.1, halo=False), dims, K, lr=0.5, flags=128)
    with g:
        g.train_epoch()
        oracle_step(g, ref, TOL)
        before, first = [g.get_params(k) for k in range(K)], [g.get_grads(k) for k in range(K)]
        g.debug_expire_wait(1)
        g.train_epoch(wait=False)
        with pytest.raises(pkg.GadError):
            g.synchronize()
        oracle_step(g, ref, TOL)
        for k in range(K):
            assert np.array_equal(g.get_params(k), before[k])
            assert rel_err(g.get_grads(k), ref.get_grads(k)) <= TOL
            w0 = dims[0] * dims[1]                      # (that is not so because the step changed nothing)
            assert rel_err(first[k][:w0], ref.get_grads(k)[:w0]) > 10 * TOL
