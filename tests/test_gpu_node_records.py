"""The nodes' query records at the sizes where they change hands (written with the preorder parents up to
2^20 nodes, gathered by a launch of their own beyond), single trees and batches, against the oracle."""

import numpy as np
import pytest

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu

HERE = 1 << 20


@pytest.mark.parametrize("n", [4097, 5000, 70001, HERE - 1, HERE, HERE + 1])
@pytest.mark.parametrize("grasp", [1, 40, None])
def test_queries(n, grasp):
    import paper_2103_15217_gb300 as etl
    parent = synth.tree_parent(n, grasp, seed=n)
    u, v = synth.lca_queries(n, 20011, seed=n)
    h = etl.lca_preprocess(dev(parent))
    assert (host(h.query(dev(u), dev(v))) == oracle.lca_offline(parent, u, v)).all()
    assert h.status() == 0


@pytest.mark.parametrize("sizes", [(1, 31, 4097, 2), (HERE // 2, HERE // 2), (HERE // 2, 1, HERE // 2)])
def test_batches(sizes):
    import paper_2103_15217_gb300 as etl
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    trees = [synth.tree_parent(n, 64, seed=i + 1) for i, n in enumerate(sizes)]
    q = [synth.lca_queries(n, 3001, seed=i + 1) for i, n in enumerate(sizes)]
    inst = np.repeat(np.arange(len(sizes)), 3001).astype(np.int32)
    u, v = (np.concatenate([p[j] for p in q]).astype(np.int32) for j in (0, 1))
    h = etl.lca_preprocess_batch(dev(np.concatenate(trees).astype(np.int32)), dev(off), max(sizes))
    want = np.concatenate([oracle.lca_offline(t, a, b) for t, (a, b) in zip(trees, q)])
    assert (host(h.query_batch(dev(inst), dev(u), dev(v))) == want).all()
    assert h.status() == 0
