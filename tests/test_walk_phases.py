"""The forms of the ranking walk are timed under names of their own, each with the bytes it moves per element
in the benchmark's roofline."""

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_bytes_per_launch():
    import numpy as np
    trees = [dict(n=1 << 24, u=np.zeros(4, np.int32)) for _ in range(3)]
    graphs = [dict(n=1 << 22, m=(1 << 25) - 1)] * 2
    assert bench.algorithmic_bytes_per_launch("rank.walk0_in_place", trees, graphs) == 8 * 2 * (1 << 24)
    assert bench.algorithmic_bytes_per_launch("rank.walk0_list", trees, graphs) == 8 * (2 * (1 << 22) - 1)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n,phase", [("list", 15361, "rank.walk0_list"), ("list", 12582912, "rank.walk0_list"),
                                          ("list", 12582913, "rank.walk0_in_place"), ("tree", 8193, "rank.walk0"),
                                          ("tree", 1 << 21, "rank.walk0"), ("tree", (1 << 21) + 1, "rank.walk0_in_place")])
def test_names(kind, n, phase):
    import torch

    import paper_2103_15217_gb300 as etl
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    etl.profile_reset()
    etl.profile_enable(True)
    try:
        if kind == "tree":
            h = etl.lca_preprocess(v - 1)
            assert h.status() == 0
        else:
            succ = v + 1
            succ[-1] = -1
            assert torch.equal(etl.list_rank(succ, 0), v)
        got = [k for k in etl.profile_read() if k.startswith("rank.walk0")]
    finally:
        etl.profile_enable(False)
        etl.profile_reset()
    assert got == [phase]
