"""Bridges at the places where the connectivity pass and the forest's tour change form: graphs hooked in
one launch (up to 49152 edges) and in slices (the giant component's root found beside the compression or
after it), edge arrays that are and are not 8-byte aligned, forests of many components (each starts a tour
of its own in one list), stars (one tail for every half-edge), isolated vertices and loops. Masks and
2-edge-connected labels are unique, so they are compared exactly."""

import numpy as np
import pytest
import torch

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu

AT_ONCE = 98304


def many_components(n, m, size, seed):
    """Random edges inside consecutive groups of `size` vertices, loops and parallel edges included."""
    rng = np.random.default_rng(seed)
    g = rng.integers(0, -(-n // size), m)
    lo = g * size
    hi = np.minimum(lo + size, n)
    return np.stack([lo + rng.integers(0, hi - lo), lo + rng.integers(0, hi - lo)], 1).astype(np.int32)


def star(n, seed):
    rng = np.random.default_rng(seed)
    e = np.stack([np.full(n - 1, n // 2), np.delete(np.arange(n), n // 2)], 1)
    extra = rng.integers(0, n, (n // 3, 2))
    return rng.permutation(np.concatenate([e, extra])).astype(np.int32)


CASES = [(f"easy {m}", lambda m=m: (20000, synth.easy_graph(20000, m, seed=m))) for a in (AT_ONCE // 2, AT_ONCE) for m in (a - 1, a, a + 1)] + \
        [(f"random {n}", lambda n=n: (n, synth.easy_graph(n, 2 * n, seed=n))) for n in (1 << 17, (1 << 17) + 1, 1 << 18, (1 << 18) + 1)] + \
        [(f"paths {n}", lambda n=n: (n, synth.hard_graph(n, n, n // 100, seed=n))) for n in (1 << 17, (1 << 18) + 1)] + \
        [(f"groups of {s}", lambda s=s: (50001, many_components(50001, 60000, s, s))) for s in (1, 2, 3, 33, 1000)] + \
        [("large groups", lambda: (300000, many_components(300000, 500000, 5, 7))),
         ("star", lambda: (40001, star(40001, 1))), ("large star", lambda: (200000, star(200000, 2))),
         ("two vertices", lambda: (2, np.array([[1, 0]], np.int32))), ("loop", lambda: (1, np.array([[0, 0]], np.int32))),
         ("loops", lambda: (5, np.array([[2, 2], [4, 4]], np.int32)))]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_masks_and_labels(name, make):
    import paper_2103_15217_gb300 as etl
    n, e = make()
    m = e.shape[0]
    want = oracle.bridges_dfs(n, e)
    flat = torch.empty(2 * m + 1, dtype=torch.int32, device="cuda")
    flat[1:] = dev(e).flatten()
    for edges in (dev(e), flat[1:].view(m, 2)):
        st = etl.new_status()
        assert (host(etl.find_bridges(edges, n, status=st)) == want).all()
        assert int(st) == 0
        assert (host(etl.find_bridges(edges, n, method="hybrid")) == want).all()
        assert (host(etl.two_edge_cc(edges, n)) == oracle.two_edge_cc(n, e)).all()
