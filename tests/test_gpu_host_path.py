"""The host side of the calls: epochs replayed as a graph on any stream and with dropout, results copied through the pinned
ring at its edges."""
import numpy as np
import pytest

import __graft_entry__ as entry
from conftest import small_random_case, rel_err
from test_gpu_parity import make_pair, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


@pytest.mark.parametrize("own_stream", [False, True])
def test_dropout_epochs_replayed_follow_the_epoch_counter(own_stream):
    """Epochs with dropout are replayed too (the mask's epoch is a device counter): the same masks as the oracle's, launch by
    launch and replayed, local and full epochs in turn, and after the counter has been set."""
    import torch
    case = small_random_case(71, n=300, K=3, p=0.03)
    kw = dict(lr=0.1, dropout=0.5)
    if own_stream:
        kw["stream"] = torch.cuda.Stream()
    g, ref, _ = make_pair(case, (20, 24, 6), 71, **kw)
    h, _, _ = make_pair(case, (20, 24, 6), 71, flags=8, **kw)
    with g, h:
        for step in range(4):
            lg, lr = g.train_epoch(), ref.train_epoch()
            assert np.max(np.abs(lg - lr)) <= 1e-4
            assert np.array_equal(lg, h.train_epoch())
        assert rel_err(g.get_params(0), ref.get_params(0)) <= TOL
        for _ in range(2):
            assert np.array_equal(g.train_epoch_local(), h.train_epoch_local())
        assert g.epoch == 6
        g.epoch = h.epoch = 2
        assert np.array_equal(g.train_epoch(), h.train_epoch())
        assert np.array_equal(g.get_params(1), h.get_params(1))


@pytest.mark.parametrize("n,classes", [(3, 1), (4096, 64), (4097, 64), (20011, 67), (65536, 64), (150011, 67)])
def test_forward_copies_every_row_through_the_ring(n, classes):
    """Less than a slot, slots of several sizes, whole and ragged, one round of the ring and several; rows that no
    subgraph owns are zero."""
    rowptr = np.arange(n + 1, dtype=np.int64)
    col = np.arange(n, dtype=np.int32)                 # self-loops only: A~ is the identity
    core = np.arange(n - 1, dtype=np.int32)            # the last node belongs to no subgraph
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 4)).astype(np.float32)
    W = rng.standard_normal((4, classes)).astype(np.float32)
    b = rng.standard_normal(classes).astype(np.float32)
    import paper_2110_02987_b200 as pkg
    z = np.zeros(2, np.int64)
    with pkg.Gad(n, rowptr, col, np.array([0, n - 1]), core, z, np.empty(0, np.int32), X, np.zeros(n, np.int32), np.zeros(n, np.uint8),
                 (4, classes), init_params=np.concatenate([W.ravel(), b])) as g:
        for _ in range(2):
            out = g.forward()
            assert not out[n - 1].any()
            assert rel_err(out[:-1], (X.astype(np.float64) @ W + b)[:-1]) <= 1e-5
