"""The list ranker's forms at the sizes where one gives way to the next: one CTA (up to 15360
elements), separate records with one and with two upper levels, records in place (beyond 12,582,912
elements, 2^21 tree nodes), for trees in 4-byte slots up to 2^25 nodes. A list built from a permutation has rank[perm[i]] = i, so the results are compared exactly."""

import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

TOP = 15360
IN_PLACE = (96 << 20) // 8  # the longest list with separate records


def make_list(n, kind, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "random":
        order = torch.randperm(n, generator=g, device="cuda", dtype=torch.int64)
    elif kind == "identity":
        order = torch.arange(n, device="cuda")
    else:  # evens downwards, then odds
        order = torch.cat([torch.arange(0, n, 2, device="cuda").flip(0), torch.arange(1, n, 2, device="cuda")])
    succ = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    succ[order[:-1]] = order[1:].int()
    rank = torch.empty(n, dtype=torch.int32, device="cuda")
    rank[order] = torch.arange(n, dtype=torch.int32, device="cuda")
    return succ, int(order[0]), rank, order


@pytest.mark.parametrize("n", [1, 2, 5, 1023, 1025, 4095, 4097, TOP - 1, TOP, TOP + 1, 2 * TOP + 1, (1 << 15) + 1,
                               (1 << 17) + 1, (1 << 18) - 1, (1 << 20) + 1, IN_PLACE, IN_PLACE + 1, (1 << 24) + 3])
@pytest.mark.parametrize("kind", ["random", "identity", "evens"])
def test_lists(n, kind):
    import paper_2103_15217_gb300 as etl
    succ, head, want, _ = make_list(n, kind)
    keep = succ.clone()
    st = etl.new_status()
    assert torch.equal(etl.list_rank(succ, head, status=st), want)
    assert int(st) == 0
    assert torch.equal(succ, keep)


@pytest.mark.parametrize("n", [TOP, 1 << 18, IN_PLACE + 1])
def test_ranks_over_the_list_itself(n):
    # the C entry point with rank == succ
    import paper_2103_15217_gb300 as etl
    lib = etl.load_library()
    succ, head, want, _ = make_list(n, "random", 2)
    p = ctypes.c_void_p(succ.data_ptr())
    assert lib.etl_list_rank(p, n, head, p, None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    assert torch.equal(succ, want)


@pytest.mark.parametrize("n", [1000, TOP, 1 << 18, IN_PLACE + 1])
@pytest.mark.parametrize("fault", ["two lists", "rho", "cycle", "past the end", "off marker", "below -1"])
def test_malformed_lists_end_with_a_status(n, fault):
    import paper_2103_15217_gb300 as etl
    succ, head, _, order = make_list(n, "random", 3)
    a, mid, tail = (int(order[i]) for i in (n // 3, n // 2, n - 1))
    at, to = {"two lists": (mid, -1), "rho": (tail, a), "cycle": (tail, head), "past the end": (mid, n),
              "off marker": (tail, 0x7ffffffe), "below -1": (mid, -7)}[fault]
    succ[at] = to
    st = etl.new_status()
    etl.list_rank(succ, head, status=st)
    assert int(st) != 0


@pytest.mark.parametrize("n,grasp", [(n, g) for n in (TOP // 2, TOP // 2 + 1, (1 << 20) + 3, 1 << 21, (1 << 21) + 1, (1 << 22) + 1)
                                     for g in (1, 3, 1024)] + [((1 << 25) + 1, 3)])
def test_trees(n, grasp):
    # the tour of a tree by the grasp model: depth, size and preorder from the definition
    import oracle
    import synth
    import paper_2103_15217_gb300 as etl
    parent = synth.tree_parent(n, grasp, seed=n)
    h = etl.lca_preprocess(torch.from_numpy(parent).cuda())
    got = {k: v.cpu().numpy() for k, v in h.arrays().items()}
    assert h.status() == 0
    pre, depth, size, _ = oracle.tree_tour(parent)
    assert (got["pre"] == pre).all() and (got["depth"] == depth).all() and (got["size"] == size).all()
    assert (got["order"][pre] == range(n)).all()
