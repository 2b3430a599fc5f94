"""Graphs whose vertices and edges are listed along a path or a cycle, in order or from the end: every edge of
the path is a bridge, none of the cycle. The hooking must not build one long chain of them that a late edge
climbs alone (tens of milliseconds where the shuffled path takes 0.3), so the time is compared with the
same path's in random order on permuted labels: ten times that is allowed, a chain costs thirty and more."""

import statistics

import pytest
import torch

pytestmark = pytest.mark.gpu


def edges_of(kind, n):
    v = torch.arange(n, device="cuda", dtype=torch.int32)
    e = torch.stack([v[:-1], v[1:]], 1)
    if kind == "from the end":
        e = e.flip(0).flip(1)
    elif kind == "cycle":
        e = torch.stack([v, torch.roll(v, -1)], 1)
    elif kind == "shuffled":
        g = torch.Generator(device="cuda").manual_seed(n)
        e = torch.randperm(n, generator=g, device="cuda").int()[e.long()]
        e = e[torch.randperm(n - 1, generator=g, device="cuda")]
    return e.contiguous()


@pytest.mark.parametrize("n", [2, 3, 300, 16384, (1 << 17) + 1, 1 << 20])
@pytest.mark.parametrize("kind", ["in order", "from the end", "cycle", "shuffled"])
def test_masks(kind, n):
    import paper_2103_15217_gb300 as etl
    e = edges_of(kind, n)
    want = 0 if kind == "cycle" else 1  # n = 2: two parallel edges are a cycle
    assert bool((etl.find_bridges(e, n) == want).all())
    if n <= 16384:
        label = etl.two_edge_cc(e, n)
        v = torch.arange(n, device="cuda", dtype=torch.int32)
        assert torch.equal(label, torch.zeros_like(v) if kind == "cycle" else v)


def time_of(etl, e, n):
    ts = []
    for i in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        etl.find_bridges(e, n)
        b.record()
        b.synchronize()
        if i >= 2:
            ts.append(a.elapsed_time(b))
    return statistics.median(ts)


@pytest.mark.parametrize("kind,n", [("in order", 1 << 20), ("from the end", 1 << 20), ("cycle", 1 << 20), ("cycle", 1 << 14)])
def test_no_long_chain(kind, n):
    import paper_2103_15217_gb300 as etl
    usual = time_of(etl, edges_of("shuffled", n), n)
    assert time_of(etl, edges_of(kind, n), n) < 10 * usual
