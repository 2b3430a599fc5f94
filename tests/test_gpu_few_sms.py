"""Streams that have only some of the device's SMs (a green context): trees whose preprocessing includes the
cooperative sort of long families, with and without such families, and bridges, eagerly and from a captured
graph."""

import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        if not hasattr(cu, name) or getattr(cu, name)(*args) != 0:
            pytest.skip(f"{name} is not available")

    d, count = ctypes.c_int(), ctypes.c_uint(1)
    whole, part, rest = (ctypes.create_string_buffer(512) for _ in range(3))
    desc, ctx, s = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    call("cuDeviceGet", ctypes.byref(d), torch.cuda.current_device())
    call("cuDeviceGetDevResource", d, whole, 1)  # the SMs
    call("cuDevSmResourceSplitByCount", part, ctypes.byref(count), whole, rest, 0, 16)
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
    call("cuGreenCtxCreate", ctypes.byref(ctx), desc, d, 1)  # 1: its own default stream
    call("cuGreenCtxStreamCreate", ctypes.byref(s), ctx, 1, 0)  # 1: non-blocking
    yield torch.cuda.ExternalStream(s.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(s)
    cu.cuGreenCtxDestroy(ctx)


def hub_tree(n, hubs, seed):
    rng = np.random.default_rng(seed)
    par = rng.integers(0, np.minimum(np.arange(1, n), hubs))
    perm = rng.permutation(n)
    out = np.full(n, -1, np.int32)
    out[perm[1:]] = perm[par]
    return out


@pytest.mark.parametrize("kind,n", [("random", 70001), ("random", 1 << 20), ("hubs", 9000), ("hubs", 1 << 20)])
def test_trees(stream, kind, n):
    import paper_2103_15217_gb300 as etl
    parent = synth.tree_parent(n, None, seed=n) if kind == "random" else hub_tree(n, 50, n)
    P = dev(parent)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        h = etl.lca_preprocess(P)
        pre = host(h.arrays()["pre"])
        assert h.status() == 0
    assert (pre == oracle.tree_tour(parent)[0]).all()


def test_bridges(stream):
    import paper_2103_15217_gb300 as etl
    e = synth.hard_graph(200000, 300000, 3000, seed=1)
    E = dev(e)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        got = host(etl.find_bridges(E, 200000))
    assert (got == oracle.bridges_dfs(200000, e)).all()


def test_captured(stream):
    import paper_2103_15217_gb300 as etl
    n = 1 << 20
    parent = hub_tree(n, 50, 3)
    P, u = dev(parent), dev(np.arange(n, dtype=np.int32))
    out = torch.full((n,), -5, dtype=torch.int32, device="cuda")
    ws = etl.new_workspace(etl.workspace_size("lca_preprocess", n))
    v = u.flip(0).contiguous()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):  # refused if the grid does not fit the stream's SMs, which a capture would not show
        h = etl.lca_preprocess(P)
        assert h.status() == 0
        h.free()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        h = etl.lca_preprocess(P, workspace=ws)
        h.query(u, v, out=out)
    with torch.cuda.stream(stream):
        g.replay()
    torch.cuda.synchronize()
    assert h.status() == 0
    assert (host(out) == oracle.lca_offline(parent, host(u), host(v))).all()
    h.free()
