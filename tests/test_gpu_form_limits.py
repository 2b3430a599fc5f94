"""Limits between forms that single small trees no longer reach, and the continuation of a full sublist in the
walk in place: tours of 15360 brackets and more (one block ranks up to that) as batches and with full tables,
query records of trees just above the one-launch size, and lists that hold all of the walk's starting points
back to their end, so that the head's walk fills one sublist after another by itself."""

import numpy as np
import pytest
import torch

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7679, 7680, 7681])
@pytest.mark.parametrize("grasp", [1, 3, None])
def test_one_block_ranking_of_a_batch(n, grasp):
    import paper_2103_15217_gb300 as etl
    sizes = [n - 1000, 1, 999]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    trees = [synth.tree_parent(k, grasp, seed=k) for k in sizes]
    h = etl.lca_preprocess_batch(dev(np.concatenate(trees)), dev(off), max(sizes))
    arr = {k: host(t) for k, t in h.arrays().items()}
    assert h.status() == 0
    for i, t in enumerate(trees):
        pre, depth, size, _ = oracle.tree_tour(t)
        at = slice(off[i], off[i + 1])
        assert (arr["pre"][at] - off[i] == pre).all() and (arr["depth"][at] == depth).all() and (arr["size"][at] == size).all()


@pytest.mark.parametrize("n", [1, 2, 7679, 7680, 7681, 8192, 8193])
@pytest.mark.parametrize("grasp", [1, 3, None])
def test_one_block_ranking_with_full_tables(n, grasp):
    import paper_2103_15217_gb300 as etl
    old = etl.tune_get()["rmq_blocked"]
    parent = synth.tree_parent(n, grasp, seed=n)
    u, v = synth.lca_queries(n, n + 5, seed=n)
    try:
        etl.tune_set(rmq_blocked=0)
        h = etl.lca_preprocess(dev(parent))
        out = host(h.query(dev(u), dev(v)))
        arr = {k: host(t) for k, t in h.arrays().items()}
        assert h.status() == 0
    finally:
        etl.tune_set(rmq_blocked=old)
    pre, depth, size, _ = oracle.tree_tour(parent)
    assert (arr["pre"] == pre).all() and (arr["depth"] == depth).all() and (arr["size"] == size).all()
    assert (out == oracle.lca_offline(parent, u, v)).all()


@pytest.mark.parametrize("n", [8193, 8223, 8224, 8225])  # last block of 32 with one entry, 31, all and one
@pytest.mark.parametrize("grasp", [1, 40, None])
def test_records_of_small_trees(n, grasp):
    import paper_2103_15217_gb300 as etl
    parent = synth.tree_parent(n, grasp, seed=n)
    u, v = synth.lca_queries(n, 20011, seed=n)
    h = etl.lca_preprocess(dev(parent))
    assert (host(h.query(dev(u), dev(v))) == oracle.lca_offline(parent, u, v)).all()
    assert h.status() == 0


def starts(length):
    """Where the walk in place may open a sublist: floor(frac(w * golden ratio) * length) for w < length / 3."""
    w = np.arange(1, length // 3 + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
    hi, lo, n = w >> np.uint64(32), w & np.uint64(0xffffffff), np.uint64(length)
    return ((hi * n + ((lo * n) >> np.uint64(32))) >> np.uint64(32)).astype(np.int64)


FREE = 300_000  # elements before the first one a sublist may start at: 73 sublists of 4095 or 4096


def test_full_sublists_of_a_list():
    import paper_2103_15217_gb300 as etl
    n = 12582913
    taken = np.zeros(n, bool)
    taken[starts(n)] = True
    rng = np.random.default_rng(1)
    first = rng.choice(np.flatnonzero(~taken), FREE, replace=False)
    taken[:] = True
    taken[first] = False
    order = dev(np.concatenate([first, rng.permutation(np.flatnonzero(taken))]).astype(np.int32)).long()
    succ = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    succ[order[:-1]] = order[1:].int()
    st = etl.new_status()
    rank = etl.list_rank(succ, int(order[0]), status=st)
    assert int(st) == 0
    assert torch.equal(rank[order], torch.arange(n, dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("n", [(1 << 21) + 1, (1 << 25) + 1])
def test_full_sublists_of_a_tour(n):
    # a path whose first nodes' opening brackets are no starting points; 4-byte slots (sublists of 30 brackets)
    # and 8-byte ones (of 4096)
    import paper_2103_15217_gb300 as etl
    taken = np.zeros(2 * n, bool)
    taken[starts(2 * n)] = True
    free = np.flatnonzero(~taken[::2])
    assert free.size > FREE
    rng = np.random.default_rng(2)
    first = rng.choice(free, FREE, replace=False)
    rest = np.ones(n, bool)
    rest[first] = False
    path = dev(np.concatenate([first, rng.permutation(np.flatnonzero(rest))]).astype(np.int32)).long()
    parent = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    parent[path[1:]] = path[:-1].int()
    h = etl.lca_preprocess(parent)
    arr = h.arrays()
    assert h.status() == 0
    at = torch.arange(n, dtype=torch.int32, device="cuda")
    assert torch.equal(arr["pre"][path], at) and torch.equal(arr["depth"][path], at)
    assert torch.equal(arr["size"][path], n - at) and torch.equal(arr["order"].long(), path)
