"""Ranks written over part of the list: rank = succ + d for shifts to both sides, on both sides of the longest
list whose records are kept apart (12,582,912 elements; longer ones are ranked in place). A list built from a
permutation has rank[perm[i]] = i, so the results are compared exactly."""

import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

IN_PLACE = (96 << 20) // 8  # the longest list with separate records


def overlapping(n, shift, seed):
    """(succ, rank) views of one buffer, rank = succ + shift, the head and the right ranks."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    order = torch.randperm(n, generator=g, device="cuda")
    buf = torch.full((n + abs(shift),), -5, dtype=torch.int32, device="cuda")
    succ, rank = buf[max(0, -shift):][:n], buf[max(0, shift):][:n]
    succ[order[:-1]] = order[1:].int()
    succ[order[-1]] = -1
    want = torch.empty(n, dtype=torch.int32, device="cuda")
    want[order] = torch.arange(n, dtype=torch.int32, device="cuda")
    return succ, rank, int(order[0]), want


def pointer(t):
    return ctypes.c_void_p(t.data_ptr())


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("n", [1000, 15360, 15361, 1 << 18, IN_PLACE, IN_PLACE + 1, 1 << 24])
@pytest.mark.parametrize("shift", [1, -1, 1000, -1000])
def test_shifted_ranks(n, shift):
    import paper_2103_15217_gb300 as etl
    lib = etl.load_library()
    succ, rank, head, want = overlapping(n, shift, n + shift)
    st = etl.new_status()
    assert lib.etl_list_rank(pointer(succ), n, head, pointer(rank), pointer(st), stream()) == 0
    assert int(st) == 0
    assert torch.equal(rank, want)


@pytest.mark.parametrize("n", [1000, 1 << 18])
@pytest.mark.parametrize("shift", [0, 1, -1000])
def test_shifted_ranks_without_allocation(n, shift):
    import paper_2103_15217_gb300 as etl
    lib = etl.load_library()
    succ, rank, head, want = overlapping(n, shift, n + shift)
    st = etl.new_status()
    assert lib.etl_list_rank_static(pointer(succ), n, head, pointer(rank), pointer(st), stream()) == 0
    assert int(st) == 0
    assert torch.equal(rank, want)


@pytest.mark.parametrize("n", [1, 1000, 15361, IN_PLACE, IN_PLACE + 1])
@pytest.mark.parametrize("shift", [0, 1, -1000, None])
def test_workspace_covers_every_overlap(n, shift):
    # the reported size is enough however the arrays lie; where they overlap but are not the same, and the
    # caller gives no status word, it is needed to the byte (256 of it are room to align the buffer, which is
    # aligned here)
    import paper_2103_15217_gb300 as etl
    lib = etl.load_library()
    succ, rank, head, want = overlapping(n, n + 8 if shift is None else shift, n)
    need = etl.workspace_size("list_rank", n)
    ws = etl.new_workspace(need)
    assert ws.data_ptr() % 256 == 0
    st = etl.new_status()
    call = lambda size, st: lib.etl_list_rank_ws(pointer(succ), n, head, pointer(rank), st, pointer(ws), size, stream())
    if shift and abs(shift) < n:
        assert call(need - 257, None) == 2  # ETL_ENOMEM
        succ, rank, head, want = overlapping(n, shift, n)
    a0 = etl.alloc_count()
    assert call(need, None) == 0
    assert torch.equal(rank, want)
    succ, rank, head, want = overlapping(n, n + 8 if shift is None else shift, n + 1)
    assert call(need, pointer(st)) == 0
    assert etl.alloc_count() == a0
    assert int(st) == 0
    assert torch.equal(rank, want)
