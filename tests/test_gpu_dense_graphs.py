"""Many edges on few vertices, where most updates of low and high are found to change nothing by a load: two
parts with random edges inside each, joined by one bridge, with pendant vertices on both, against the oracle;
edge counts on both sides of the line (2^19 edges, 128 per tour position)."""

import numpy as np
import pytest

import oracle
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


def two_parts(n, m, seed):
    rng = np.random.default_rng(seed)
    core = n - n // 8  # the rest are pendant
    half = core // 2
    k = m - 1 - (n - core)
    side = rng.integers(0, 2, k)
    lo, size = np.where(side, half, 0), np.where(side, core - half, half)
    e = [np.stack([lo + rng.integers(0, size), lo + rng.integers(0, size)], 1), [[0, half]]]
    if n > core:
        e.append(np.stack([np.arange(core, n), rng.integers(0, core, n - core)], 1))
    e = np.concatenate(e).astype(np.int32)
    e = e[rng.permutation(m)]
    flip = rng.random(m) < 0.5
    e[flip] = e[flip][:, ::-1]
    perm = rng.permutation(n).astype(np.int32)
    return np.ascontiguousarray(perm[e])


@pytest.mark.parametrize("n,m", [(2, 1 << 19), (3, 1 << 19), (20, (1 << 19) - 1), (20, 1 << 19), (100, 1 << 21),
                                 (2000, (1 << 19) + 1), (2048, 128 * 4095 - 1), (2049, 128 * 4097), (30000, 128 * 59999)])
@pytest.mark.parametrize("blocked", [1, 0])
def test_masks(n, m, blocked):
    import paper_2103_15217_gb300 as etl
    e = two_parts(n, m, n)
    old = etl.tune_get()["rmq_blocked"]
    try:
        etl.tune_set(rmq_blocked=blocked)
        got = host(etl.find_bridges(dev(e), n))
    finally:
        etl.tune_set(rmq_blocked=old)
    want = oracle.bridges_dfs(n, e)
    assert want.sum() >= 1
    assert (got == want).all()
