"""The radix passes over long families that are out of order, in every form the tuning knobs select (tiles of
2048 or 4096 labels, equal digits found by ballots or by __match_any_sync), with few blocks and with many: trees
with one hub and with two thousand, of more than 8192 nodes (smaller ones take one launch), on both sides of
64 tiles and of 2^19 nodes. The preorder is unique, so it is compared with the oracle exactly."""

import numpy as np
import pytest

import oracle
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


def hub_tree(n, hubs, seed):
    """Node 0 the root; later nodes hang from a random one of the first `hubs` nodes; labels permuted."""
    rng = np.random.default_rng(seed)
    par = rng.integers(0, np.minimum(np.arange(1, n), hubs))
    perm = rng.permutation(n)
    out = np.full(n, -1, np.int32)
    out[perm[1:]] = perm[par]
    return out


@pytest.fixture
def restore_tuning():
    import paper_2103_15217_gb300 as etl
    old = etl.tune_get()
    yield
    etl.tune_set(sort_rounds=old["sort_rounds"], sort_ballot=old["sort_ballot"])


@pytest.mark.parametrize("rounds", [8, 16])
@pytest.mark.parametrize("ballot", [0, 1])
@pytest.mark.parametrize("n", [8193, 64 * 2048, 64 * 2048 + 1, 64 * 4096 + 1, 1 << 19, (1 << 19) + 1])
def test_forms(restore_tuning, rounds, ballot, n):
    import paper_2103_15217_gb300 as etl
    etl.tune_set(sort_rounds=rounds, sort_ballot=ballot)
    for hubs in (1, 2000 if n > 100000 else 100):
        parent = hub_tree(n, hubs, n + hubs)
        assert np.bincount(parent[parent >= 0]).max() > 32
        h = etl.lca_preprocess(dev(parent))
        arr = {k: host(t) for k, t in h.arrays().items()}
        assert h.status() == 0
        pre, depth, size, _ = oracle.tree_tour(parent)
        assert (arr["pre"] == pre).all() and (arr["depth"] == depth).all() and (arr["size"] == size).all()


@pytest.mark.parametrize("n", [33, 34, 2048, 2049, 5000])
def test_few_nodes_with_full_tables(n):
    # full tables keep small trees on this path
    import paper_2103_15217_gb300 as etl
    old = etl.tune_get()["rmq_blocked"]
    try:
        etl.tune_set(rmq_blocked=0)
        parent = hub_tree(n, 1, n)
        h = etl.lca_preprocess(dev(parent))
        pre = host(h.arrays()["pre"])
        assert h.status() == 0
    finally:
        etl.tune_set(rmq_blocked=old)
    assert (pre == oracle.tree_tour(parent)[0]).all()
