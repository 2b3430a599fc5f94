"""Children in ascending label order, whatever the family sizes: pushed lists, families that one thread
puts in order (up to 32 children) and longer ones, which take the radix sort, in one tree and in a
batch. The preorder is unique, so it is compared with the oracle exactly."""

import numpy as np
import pytest

import oracle
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


def hub_tree(n, hubs, seed):
    """Node 0 the root; later nodes hang from a random one of the first `hubs` nodes; labels permuted."""
    rng = np.random.default_rng(seed)
    par = np.full(n, -1, np.int64)
    i = np.arange(1, n)
    par[1:] = rng.integers(0, np.minimum(i, hubs))
    perm = rng.permutation(n)
    out = np.full(n, -1, np.int64)
    out[perm[1:]] = perm[par[1:]]
    return out.astype(np.int32)


@pytest.mark.parametrize("n", [2, 33, 34, 35, 300, 1024, 1025, 70001, 600000])
@pytest.mark.parametrize("hubs", [1, 2, 40, 3000])
def test_hub_trees(n, hubs):
    import paper_2103_15217_gb300 as etl
    parent = hub_tree(n, hubs, n + hubs)
    h = etl.lca_preprocess(dev(parent))
    arr = {k: host(t) for k, t in h.arrays().items()}
    assert h.status() == 0
    pre, depth, size, _ = oracle.tree_tour(parent)
    assert (arr["pre"] == pre).all() and (arr["depth"] == depth).all() and (arr["size"] == size).all()


@pytest.mark.parametrize("rounds,ballot", [(8, 1), (16, 0)])
def test_hub_batches(rounds, ballot):
    import paper_2103_15217_gb300 as etl
    old = etl.tune_get()
    try:
        etl.tune_set(sort_rounds=rounds, sort_ballot=ballot)
        trees = [hub_tree(n, hubs, n) for n, hubs in [(1, 1), (400000, 7), (34, 1), (90000, 500), (33, 2), (300000, 1)]]
        off = np.concatenate([[0], np.cumsum([len(t) for t in trees])]).astype(np.int32)
        h = etl.lca_preprocess_batch(dev(np.concatenate(trees)), dev(off), 400000)
        got = host(h.arrays()["pre"])
        assert h.status() == 0
        for i, t in enumerate(trees):
            assert (got[off[i]:off[i + 1]] - off[i] == oracle.tree_tour(t)[0]).all()
    finally:
        etl.tune_set(sort_rounds=old["sort_rounds"], sort_ballot=old["sort_ballot"])


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1, (1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("hubs", [30, 8000, 1 << 17])
def test_where_families_change_hands(n, hubs):
    test_hub_trees(n, hubs)


@pytest.mark.parametrize("k", [16, 41, 300])
def test_batches_pushed_in_parts(k):
    """From 16 trees on the labels are pushed in several parts of the list at a time."""
    import paper_2103_15217_gb300 as etl
    rng = np.random.default_rng(k)
    sizes = rng.integers(1, 3000, k)
    sizes[k // 2] = 40000
    trees = [hub_tree(int(n), int(rng.integers(1, 400)), i) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    h = etl.lca_preprocess_batch(dev(np.concatenate(trees)), dev(off), int(sizes.max()))
    got = host(h.arrays()["pre"])
    assert h.status() == 0
    for i, t in enumerate(trees):
        assert (got[off[i]:off[i + 1]] - off[i] == oracle.tree_tour(t)[0]).all()
