"""Small trees (one launch, up to 4096 nodes) around the sizes where their blocks, warps and table levels
end, against the oracle; malformed ones must end with the tree's status."""

import numpy as np
import pytest

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu

TINY = 4096


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 127, 129, 1000, 1023, 1024, 1025, 2049, TINY - 31, TINY, TINY + 1])
@pytest.mark.parametrize("grasp", [1, 5, None, "star"])
def test_trees(n, grasp):
    import paper_2103_15217_gb300 as etl
    if grasp == "star":
        parent = np.full(n, n // 2, np.int32)
        parent[n // 2] = -1
    else:
        parent = synth.tree_parent(n, grasp, seed=n)
    u, v = synth.lca_queries(n, 3 * n + 5, seed=n)
    for methods in (("rmq",), ("rmq", "inlabel", "tour_rmq")):
        h = etl.lca_preprocess(dev(parent), methods=methods)
        arr = {k: host(t) for k, t in h.arrays().items()}
        out = [host(h.query(dev(u), dev(v)))]
        if len(methods) > 1:
            out += [host(h.query_inlabel(dev(u), dev(v))), host(h.query_tour(dev(u), dev(v)))]
        assert h.status() == 0
        pre, depth, size, _ = oracle.tree_tour(parent)
        assert (arr["pre"] == pre).all() and (arr["depth"] == depth).all() and (arr["size"] == size).all()
        assert (arr["order"][pre] == np.arange(n)).all()
        want = oracle.lca_offline(parent, u, v)
        for o in out:
            assert (o == want).all()


@pytest.mark.parametrize("n", [2, 40, 1025, TINY])
@pytest.mark.parametrize("fault", ["two roots", "no root", "cycle", "past the end", "below -1", "own parent"])
def test_malformed_trees(n, fault):
    import paper_2103_15217_gb300 as etl
    parent = np.arange(-1, n - 1).astype(np.int32)
    at, to = {"two roots": (n - 1, -1), "no root": (0, n - 1), "cycle": (n // 2, n - 1), "past the end": (n - 1, n),
              "below -1": (n - 1, -2), "own parent": (n - 1, n - 1)}[fault]
    parent[at] = to
    h = etl.lca_preprocess(dev(parent))
    out = host(h.query(dev(np.zeros(5, np.int32)), dev(np.full(5, n - 1, np.int32))))
    assert h.status() == 4          # ETL_EBADTREE
    assert (out == -1).all()


@pytest.mark.parametrize("n", [5000, 8191, 8192, 8193])
@pytest.mark.parametrize("grasp", [1, 5, None, "star"])
def test_largest_trees(n, grasp):
    test_trees(n, grasp)


@pytest.mark.parametrize("n", [257, 258, 4096, 8192])
@pytest.mark.parametrize("family", [31, 64, 65, 300])
def test_families(n, family):
    """Every node has `family` children (as long as there are labels), labels permuted."""
    import paper_2103_15217_gb300 as etl
    perm = np.random.default_rng(n).permutation(n)
    parent = np.full(n, -1, np.int32)
    parent[perm[1:]] = perm[(np.arange(1, n) - 1) // family]
    h = etl.lca_preprocess(dev(parent))
    pre, depth, size, _ = oracle.tree_tour(parent)
    arr = {k: host(t) for k, t in h.arrays().items()}
    assert h.status() == 0
    assert (arr["pre"] == pre).all() and (arr["depth"] == depth).all() and (arr["size"] == size).all()


@pytest.mark.parametrize("fault", ["two roots", "no root", "cycle", "past the end", "below -1", "own parent"])
def test_malformed_largest(fault):
    test_malformed_trees(8192, fault)
