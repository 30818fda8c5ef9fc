"""What the library is timed on: training epochs, inference, input streaming, importance weights and augmentation, through the
public entry points of ``paper_2110_02987_b200``, from the smallest graphs to ones whose operands exceed the L2 cache.

Every case is a dict of plain values.  ``kind`` says which call it is:

  train     one ``Gad.train_epoch`` (Algorithm 2: forward, loss, backward, importance weights, update and consensus) and the new
            parameters handed on with ``export_params``.  ``wait`` = the losses of every epoch are read (`loss = g.train_epoch()`),
            otherwise epochs are enqueued and the losses land in pinned memory.  ``own_stream`` = the context runs on a stream
            of its own instead of torch's default one.
  stream    the same behind ``set_inputs`` with new features and labels from pinned host memory in every step
  forward   ``Gad.forward``: logits of every node on the host
  weights   ``Gad.subgraph_weights`` in the pairwise form (zeta_mode 1)
  augment   ``Augmenter.run``: the replication-node lists of a partition (Algorithm 1)

Graphs: ``power`` has power-law expected degrees and planted communities, ``blocks`` uniform degrees inside equal communities;
subgraphs are contiguous blocks of nodes along the communities, their replicated nodes the best-connected one-hop neighbours.
They are drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

import paper_2110_02987_b200 as gad

# A step long enough for the gradients to show in the parameters that come back.
LR = 0.5

_TRAIN = dict(kind="train", graph="power", halo=0.05, gemm_mode=0, dropout=0.0, wait=False, own_stream=True)


def _case(**kw):
    c = dict(_TRAIN)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest job: 2000 nodes, narrow layers; launches and the wait for the losses are all there is
        _case(name="tiny_epoch", n=2000, degree=12.0, graph="blocks", communities=4, K=4, dims="32-16-4", wait=True, own_stream=False),
        # a citation graph with bag-of-words features: few nodes, an odd number of very wide inputs, three layers
        _case(name="citation_small", n=2708, degree=4.0, communities=7, K=4, dims="1433-128-128-7", wait=True, own_stream=False),
        # a middling citation graph trained with dropout, three classes
        _case(name="citation_dropout", n=19717, degree=4.5, communities=16, K=8, dims="500-256-3", dropout=0.5, wait=True, own_stream=True),
        # the ordinary job: a power-law graph of 100 000 nodes, one hidden layer, epochs enqueued back to back
        _case(name="ordinary_epoch", n=100000, degree=20.0, communities=16, K=8, halo=0.10, dims="128-128-16"),
        # many partitions of an image graph and a deep net: every subgraph is small (1785 core nodes)
        _case(name="many_subgraphs", n=89250, degree=20.0, communities=50, K=50, dims="500-128-128-128-7", wait=True, own_stream=False),
        # dense communities with wide features (posts of a discussion site): the aggregation is nearly everything
        _case(name="dense_communities", n=60000, degree=300.0, graph="blocks", communities=16, K=8, dims="602-256-41"),
        # the largest: a product graph, three layers of 256; one subgraph's operand exceeds the L2 cache
        _case(name="large_epoch", n=500000, degree=40.0, communities=48, K=4, dims="100-256-256-47"),
        # the same net in the reduced-precision mode on more and smaller subgraphs
        _case(name="reduced_precision", n=200000, degree=40.0, communities=48, K=16, dims="100-256-256-47", gemm_mode=1),
        # features and labels that change from step to step, uploaded from pinned memory
        _case(name="streamed_inputs", kind="stream", n=100000, degree=20.0, communities=16, K=8, halo=0.10, dims="128-128-16"),
        # inference over all nodes, logits to the host
        _case(name="inference", kind="forward", n=100000, degree=20.0, communities=16, K=8, halo=0.10, dims="128-256-40", own_stream=False),
        # importance weights from all pairs of nodes of a subgraph
        _case(name="pairwise_weights", kind="weights", n=50000, degree=20.0, communities=16, K=8, dims="128-128-16", own_stream=False),
        # replication nodes by random walks for eight core sets of the ordinary graph
        _case(name="augmentation", kind="augment", n=100000, degree=20.0, communities=16, K=8, dims="128-128-16", own_stream=False),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["train"] * 11 + ["stream"] * 2 + ["forward"] * 3 + ["weights"] * 1 + ["augment"] * 2)
    c = _case(kind=kind, graph=rng.choice(["power", "power", "blocks"]))
    c["n"] = int(_log_uniform(rng, 1500, 60000 if kind == "weights" else 100000 if kind == "augment" else 400000))
    c["degree"] = round(_log_uniform(rng, 4.0, 40.0 if kind == "augment" else 300.0), 2)
    layers = rng.choice([2, 2, 3, 3, 4])
    hidden = int(_log_uniform(rng, 16, 512))
    first = int(_log_uniform(rng, 24, 1433))
    c["dims"] = "-".join(str(d) for d in [first] + [hidden] * (layers - 1) + [rng.randint(2, 64)])
    if kind in ("train", "stream", "forward"):
        c["gemm_mode"] = 1 if rng.random() < 0.15 else 0
    if kind == "train":
        c["dropout"] = rng.choice([0.0, 0.0, 0.5])
    c["wait"], c["own_stream"] = rng.random() < 0.5, rng.random() < 0.5
    c["K"] = max(2, min(50, int(_log_uniform(rng, 2, 50)), c["n"] // 400))
    c["communities"] = max(c["K"], rng.randint(4, 50))
    c["halo"] = rng.choice([0.05, 0.10])
    # no more entries, features or multiply-adds than the largest listed cases have
    while (c["n"] * c["degree"] > 18e6 or c["n"] * first > 48e6 or work(c)["flops"] > 3e11) and c["n"] > 1500:
        c["n"] = max(1500, int(c["n"] * 0.8))
        c["K"] = max(2, min(c["K"], c["n"] // 400))
    return c


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("-"))


def _intra(case):
    """Share of the edges drawn inside one community."""
    return 0.8 if case["graph"] == "blocks" else 0.7


def _graph(case, gen):
    """Undirected graph with self-loops as CSR (rowptr int64, col int32, ascending), on the GPU; nodes are numbered community by
    community."""
    n, m, nc = case["n"], int(case["n"] * case["degree"] / 2), case["communities"]
    dev = gen.device

    def uniform(k):
        return torch.rand(k, generator=gen, device=dev, dtype=torch.float64)

    bounds = torch.linspace(0, n, nc + 1, device=dev, dtype=torch.float64).round().to(torch.int64)
    if case["graph"] == "power":
        w = (torch.arange(n, device=dev, dtype=torch.float64) + 10.0) ** (-1.0 / 1.1)
        w = w[torch.randperm(n, generator=gen, device=dev)]
        w = w * (case["degree"] * n / w.sum())
        w = torch.clamp(w, max=float(w.sum().sqrt()))       # pair probabilities stay below one
    else:
        w = torch.ones(n, device=dev, dtype=torch.float64)
    cdf = torch.cumsum(w, 0)
    u = torch.searchsorted(cdf, uniform(m) * cdf[-1]).clamp_(max=n - 1)
    start = torch.cat([torch.zeros(1, device=dev, dtype=torch.float64), cdf])
    comm = (torch.searchsorted(bounds, u, right=True) - 1).clamp_(0, nc - 1)
    lo, hi = start[bounds[comm]], start[bounds[comm + 1]]
    inside = uniform(m) < _intra(case)
    r = uniform(m)
    v = torch.searchsorted(cdf, torch.where(inside, lo + r * (hi - lo), r * cdf[-1])).clamp_(max=n - 1)
    keep = u != v
    u, v = u[keep], v[keep]
    loop = torch.arange(n, device=dev, dtype=torch.int64)
    key = torch.unique(torch.cat([u * n + v, v * n + u, loop * n + loop]))
    row = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, device=dev, dtype=torch.int64)
    rowptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rowptr, (key - row * n).to(torch.int32), row


def _halos(case, rowptr, col, row):
    """Replicated nodes of every block: its outside neighbours by descending degree, at most `halo` times the block's size."""
    n, K = case["n"], case["K"]
    size = -(-n // K)
    c64 = col.to(torch.int64)
    part = torch.div(row, size, rounding_mode="floor")
    cross = part != torch.div(c64, size, rounding_mode="floor")
    cand = torch.unique(part[cross] * n + c64[cross])
    deg = torch.diff(rowptr)
    top = int(deg.max()) + 1
    p = torch.div(cand, n, rounding_mode="floor")
    node = cand - p * n
    order = torch.argsort((p * top + (top - 1 - deg[node])) * n + node)
    p, node = p[order], node[order]
    count = torch.bincount(p, minlength=K)
    first = torch.cumsum(count, 0) - count
    keep = torch.arange(p.numel(), device=p.device) - first[p] < math.ceil(case["halo"] * size)
    return torch.bincount(p[keep], minlength=K).cpu().numpy(), node[keep].to(torch.int32).cpu().numpy()


def prepare(case, seed):
    """The graph, features, labels and split as host arrays and the context (or the augmenter) a program keeps."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, K, dims = case["n"], case["K"], _dims(case)
    rowptr_d, col_d, row = _graph(case, gen)
    rowptr, col = rowptr_d.cpu().numpy(), col_d.cpu().numpy()
    size = -(-n // K)
    core = [np.arange(k * size, min((k + 1) * size, n), dtype=np.int32) for k in range(K)]
    state = dict(kind=case["kind"], wait=case["wait"], seed=seed)
    if case["kind"] == "augment":
        state.update(aug=gad.Augmenter(n, rowptr, col), cores=core)
        return state
    halo_count, halo = _halos(case, rowptr_d, col_d, row)
    core_ptr, halo_ptr = np.zeros(K + 1, np.int64), np.zeros(K + 1, np.int64)
    np.cumsum([len(c) for c in core], out=core_ptr[1:])
    np.cumsum(halo_count, out=halo_ptr[1:])
    # labels follow the communities, one in ten is wrong
    y = torch.arange(n, device="cuda") * case["communities"] // n
    noise = torch.rand(n, generator=gen, device="cuda") < 0.1
    y = torch.where(noise, torch.randint(0, 1 << 20, (n,), generator=gen, device="cuda"), y) % dims[-1]
    X = torch.randn(n, dims[0], generator=gen, device="cuda").cpu()
    labels = y.to(torch.int32).cpu()
    split = (torch.rand(n, generator=gen, device="cuda") * 5).to(torch.uint8).cpu().numpy()
    split = np.where(split < 3, 0, split - 2).astype(np.uint8)      # 60 / 20 / 20
    kw = dict(lr=LR, dropout=case["dropout"], seed=seed, gemm_mode=case["gemm_mode"], zeta_mode=1 if case["kind"] == "weights" else 0)
    if case["own_stream"]:
        kw["stream"] = torch.cuda.Stream()
    g = gad.Gad(n, rowptr, col, core_ptr, np.concatenate(core), halo_ptr, halo, X.numpy(), labels.numpy(), split, dims, **kw)
    state.update(g=g, params=g.new_consensus_buffer())
    if case["kind"] == "stream":
        state.update(X=X.pin_memory(), labels=labels.pin_memory())
    if not case["wait"]:
        state["loss_pinned"] = torch.zeros(K + 1, dtype=torch.float32).pin_memory()
        state["loss"] = state["loss_pinned"].numpy()
    torch.cuda.synchronize()
    return state


def run(state):
    if state["kind"] == "augment":
        halos, walks = state["aug"].run(state["cores"], 2, seed=state["seed"])
        return dict(nodes=np.concatenate(halos), sizes=np.array([len(h) for h in halos]), walks=walks)
    g = state["g"]
    if state["kind"] == "forward":
        return g.forward()
    if state["kind"] == "weights":
        zeta, w = g.subgraph_weights()
        return dict(zeta=zeta, weights=w)
    if state["kind"] == "stream":
        g.set_inputs(state["X"], state["labels"])
    if state["wait"]:
        loss = g.train_epoch()
    else:
        loss = state["loss"]
        g.train_epoch(loss_out=loss, wait=False)
    return dict(loss=loss, params=g.export_params(0, state["params"]))


def work(case):
    """Bytes of every input read once and every output written once, operations of the method on the store's expected size."""
    n, K, dims = case["n"], case["K"], _dims(case)
    rows = n * (1.0 + case["halo"])
    # entries of the augmented subgraphs: the edges inside a block, those that a replicated node brings back, self-loops
    kept = _intra(case) * min(1.0, case["communities"] / K) + (1.0 - _intra(case)) / K + 2 * case["halo"]
    nnz = n * case["degree"] * min(1.0, kept) + rows
    P = sum(dims[l] * dims[l + 1] + dims[l + 1] for l in range(len(dims) - 1))
    if case["kind"] == "augment":
        return dict(bytes=8.0 * n + 4.0 * n * (case["degree"] + 1) + 4.0 * n, flops=0.0)
    if case["kind"] == "weights":
        return dict(bytes=4.0 * rows * (dims[0] + 1) + 8.0 * K, flops=K * (rows / K) ** 2 / 2 * 2.0 * dims[0])
    transforms = [2.0 * rows * dims[l] * dims[l + 1] for l in range(len(dims) - 1)]
    spmm = [2.0 * nnz * min(dims[l], dims[l + 1]) for l in range(len(dims) - 1)]
    store = 8.0 * nnz + 4.0 * rows * dims[0]
    if case["kind"] == "forward":
        return dict(bytes=store + 4.0 * K * P + 4.0 * n * dims[-1], flops=sum(transforms) + sum(spmm))
    flops = 3 * sum(transforms) - transforms[0] + 2 * sum(spmm) - spmm[0]
    new = 4.0 * n * (dims[0] + 1) if case["kind"] == "stream" else 0.0
    return dict(bytes=store + new + 5.0 * rows + 8.0 * K * P + 4.0 * P, flops=flops)


def tolerance(case):
    if case["kind"] == "augment":
        return "exact"
    if case["gemm_mode"] == 1:      # TF32 transforms and bfloat16 gathered operands
        return {"rel": 5e-3}
    # Logits and importance weights are sums of products of 32-bit operands over up to a few thousand terms; so are the losses,
    # and the gradients, which reach the exported parameters through one step.  A hidden unit at the kink of its ReLU may fall
    # on either side.
    return {"rel": 1e-5}
