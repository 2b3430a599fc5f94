"""The work a user of the library has it do, as cases that can be timed and checked.

A case is one pass through the public entry points: preprocess a tree and answer its LCA queries,
answer queries on a tree that is already resident, rank a list, find the bridges of a graph, or do
the first and the last for a batch of small instances at once. Sizes and shapes are those of the
benchmark, the tests and the serving workload: trees by the grasp model (a node's parent is uniform
among the previous `grasp` nodes, labels permuted; grasp 0 = all previous nodes, 1 = a path), easy
graphs (random recursive spanning tree + uniform extra edges) and hard graphs (a path with short
chords and uncovered path edges).

Every output is int32 or uint8 and has one right value, so `exact` gives it by other means (pointer
doubling over the parent array, sums of random keys over the subtrees of a known spanning tree).
"""

from __future__ import annotations

import math

import torch

import paper_2103_15217_gb300 as etl

DEV = "cuda"


def listed():
    return [
        # the smallest call: one small tree of a serving set and its queries; launches and latency only
        dict(name="tree_1k", kind="tree", n=1000, grasp=0, q=1000, arrays=False, workspace=False),
        # the benchmark's small configuration, scratch and tables in a workspace the caller keeps
        dict(name="tree_64k_ws", kind="tree", n=1 << 16, grasp=0, q=1 << 16, arrays=False, workspace=True),
        # an ordinary tree of odd size; the program also takes the tour arrays (pre, depth, size, order)
        dict(name="tree_1m_arrays", kind="tree", n=1_000_003, grasp=1024, q=250_001, arrays=True, workspace=False),
        # the benchmark's large trees, one query per node: shallow, and the deepest there is
        dict(name="tree_random_16m", kind="tree", n=1 << 24, grasp=0, q=1 << 24, arrays=False, workspace=False),
        dict(name="tree_path_16m", kind="tree", n=1 << 24, grasp=1, q=1 << 24, arrays=False, workspace=False),
        # serving: the largest query batch on the largest resident tree
        dict(name="query_1m", kind="query", n=1 << 22, grasp=0, q=1 << 20),
        # the Inlabel method, odd size, one query per node
        dict(name="inlabel_4m", kind="inlabel", n=4_100_001, grasp=1024, q=4_100_001),
        # list ranking by itself, on a list in random order
        dict(name="list_rank_8m", kind="list_rank", n=8_400_007),
        # bridges of a small graph of the batched workload, and of the benchmark's two large ones
        dict(name="bridges_16k", kind="bridges", n=16_385, m=65_541, hard=False),
        dict(name="bridges_easy_4m", kind="bridges", n=1 << 22, m=(1 << 25) - 1, hard=False),
        dict(name="bridges_hard_4m", kind="bridges", n=1 << 22, m=(1 << 22) - 1 + (1 << 24), hard=True),
        # a quarter of the batched workload: trees of 2^6 .. 2^18 nodes, graphs of 2^6 .. 2^16, in one call each
        dict(name="batch_512", kind="batch", trees=512, graphs=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tree", "tree", "tree", "query", "inlabel", "list_rank", "bridges", "bridges", "batch"])
    grasp = rng.choice([0, 0, 1024, 32, 1])
    if kind == "tree":
        n = _log_int(rng, 64, 1 << 24)
        return dict(kind=kind, n=n, grasp=grasp, q=max(1, int(n * rng.uniform(0.1, 1.0))),
                    arrays=rng.random() < 0.3, workspace=rng.random() < 0.3)
    if kind == "query":
        return dict(kind=kind, n=_log_int(rng, 1 << 10, 1 << 22), grasp=grasp, q=_log_int(rng, 1 << 4, 1 << 20))
    if kind == "inlabel":
        n = _log_int(rng, 1 << 10, 1 << 23)
        return dict(kind=kind, n=n, grasp=grasp, q=max(1, int(n * rng.uniform(0.1, 1.0))))
    if kind == "list_rank":
        return dict(kind=kind, n=_log_int(rng, 1 << 10, 1 << 24))
    if kind == "bridges":
        n = _log_int(rng, 1 << 10, 1 << 22)
        return dict(kind=kind, n=n, m=int(n * rng.uniform(1.5, 7.0)), hard=rng.random() < 0.5)
    k = _log_int(rng, 16, 512)
    return dict(kind=kind, trees=k, graphs=k)


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _rand(g, n):
    return torch.rand(int(n), generator=g, device=DEV, dtype=torch.float64)


def _below(g, width):
    """Uniform integers in [0, width) per entry (width >= 1)."""
    return torch.minimum((_rand(g, width.numel()) * width).long(), width - 1)


def _offsets(sizes):
    off = torch.zeros(sizes.numel() + 1, dtype=torch.long, device=DEV)
    off[1:] = torch.cumsum(sizes, 0)
    return off


def _forest(g, sizes, grasps, permuted):
    """k trees by the grasp model, concatenated; labels permuted inside each tree where asked.
    Returns the parent array in global labels (-1 at roots), the instance of each node and the offsets."""
    off = _offsets(sizes)
    total = int(off[-1])
    inst = torch.repeat_interleave(torch.arange(sizes.numel(), device=DEV), sizes, output_size=total)
    at = torch.arange(total, device=DEV)
    i = at - off[inst]
    gr = grasps[inst]
    lo = torch.where(gr > 0, torch.clamp(i - gr, min=0), torch.zeros_like(i))
    par = lo + _below(g, torch.clamp(i - lo, min=1)) + off[inst]
    key = torch.where(permuted[inst], (_rand(g, total) * (1 << 36)).long(), i)
    label = torch.empty_like(at)
    label[torch.argsort((inst << 37) | key)] = at  # sorted by instance: labels stay inside their own
    parent = torch.empty_like(at)
    parent[label] = torch.where(i == 0, torch.full_like(i, -1), label[par])
    return parent, inst, off


def _graphs(g, n, m, hard):
    """Graphs concatenated: spanning tree (random recursive, or a path for hard ones) + extra edges
    (uniform, except that the last n / 64 labels get none, as social graphs have pendant vertices; or chords (i, i + d), 2 <= d <= 16, that jump no cut; about n / 64 path edges are cuts),
    edges shuffled inside each graph and randomly oriented. Returns edges in global ids, per edge the
    child of its tree edge (-1: extra edge), the spanning forest's parents and both offsets."""
    k = n.numel()
    parent, inst, noff = _forest(g, n, hard.long(), ~hard)
    total = parent.numel()
    child = torch.nonzero(parent >= 0).flatten()
    extra = m - (n - 1)
    ne = int(extra.sum())
    einst = torch.repeat_interleave(torch.arange(k, device=DEV), extra, output_size=ne)
    some = (n - n // 64)[einst]
    a, b = _below(g, some), _below(g, some)
    # next cut at or after each position: path edge j joins j and j + 1
    cut = _rand(g, total) < 1.0 / 64
    far = torch.where(cut, torch.arange(total, device=DEV), torch.full((total,), 1 << 40, device=DEV))
    next_cut = torch.flip(torch.cummin(torch.flip(far, [0]), 0)[0], [0])
    todo = torch.nonzero(hard[einst]).flatten()
    for _ in range(200):
        if todo.numel() == 0:
            break
        it = einst[todo]
        d = torch.minimum(2 + _below(g, torch.full_like(it, 15)), torch.clamp(n[it] - 1, min=0))
        i = _below(g, torch.clamp(n[it] - d, min=1))
        a[todo], b[todo] = i, i + d
        todo = todo[next_cut[noff[it] + i] < noff[it] + i + d]
    b[todo] = a[todo]  # no place found (tiny graphs): self-loops
    eu = torch.cat([child, a + noff[einst]])
    ev = torch.cat([parent[child], b + noff[einst]])
    ec = torch.cat([child, torch.full((ne,), -1, dtype=torch.long, device=DEV)])
    ei = torch.cat([inst[child], einst])
    order = torch.argsort((ei << 37) | (_rand(g, eu.numel()) * (1 << 36)).long())
    eu, ev, ec, ei = eu[order], ev[order], ec[order], ei[order]
    flip = _rand(g, eu.numel()) < 0.5
    edges = torch.stack([torch.where(flip, ev, eu), torch.where(flip, eu, ev)], 1)
    return dict(edges=edges, child=ec, einst=ei, parent=parent, noff=noff, eoff=_offsets(m))


def _sizes(k, lo, hi):
    """k sizes spread evenly over the logarithm of 2^lo .. 2^hi, in a mixed order: a case's own, not the seed's."""
    at = (torch.arange(k, device=DEV, dtype=torch.float64) * 0.6180339887498949) % 1.0
    return torch.exp2(lo + (hi - lo) * at).long()


def _vec(x, dtype=torch.long):
    return torch.tensor([x], dtype=dtype, device=DEV)


def _inputs(case, seed):
    """The inputs in 64 bits and global ids."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("tree", "query", "inlabel"):
        parent, _, _ = _forest(g, _vec(case["n"]), _vec(case["grasp"]), _vec(True, torch.bool))
        n = torch.full((case["q"],), case["n"], dtype=torch.long, device=DEV)
        return dict(parent=parent, u=_below(g, n), v=_below(g, n))
    if kind == "list_rank":
        order = torch.argsort((_rand(g, case["n"]) * (1 << 52)).long())
        succ = torch.empty_like(order)
        succ[order[:-1]] = order[1:]
        succ[order[-1]] = -1
        return dict(order=order, succ=succ, head=int(order[0]))
    if kind == "bridges":
        return _graphs(g, _vec(case["n"]), _vec(case["m"]), _vec(case["hard"], torch.bool))
    tn = _sizes(case["trees"], 6, 18)
    grasps = torch.tensor([1, 1024, 0], device=DEV)[torch.arange(case["trees"], device=DEV) % 3]
    parent, inst, off = _forest(g, tn, grasps, torch.ones_like(tn, dtype=torch.bool))
    u, v = off[inst] + _below(g, tn[inst]), off[inst] + _below(g, tn[inst])  # one query per node
    gn = torch.clamp(_sizes(case["graphs"], 6, 16), min=18)
    hard = torch.arange(case["graphs"], device=DEV) % 2 == 1
    return dict(parent=parent, inst=inst, off=off, tn=tn, u=u, v=v, gn=gn, graphs=_graphs(g, gn, 4 * gn, hard))


def _i32(x):
    return x.to(torch.int32).contiguous()


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("tree", "query", "inlabel"):
        st = dict(kind=kind, parent=_i32(x["parent"]), u=_i32(x["u"]), v=_i32(x["v"]))
        if kind == "tree":
            st["arrays"] = case["arrays"]
            st["ws"] = etl.new_workspace(etl.workspace_size("lca_preprocess", case["n"])) if case["workspace"] else None
        if kind == "query":
            st["handle"] = etl.lca_preprocess(st["parent"])
        return st
    if kind == "list_rank":
        return dict(kind=kind, succ=_i32(x["succ"]), head=x["head"])
    if kind == "bridges":
        return dict(kind=kind, edges=_i32(x["edges"]), n=case["n"])
    gr = x["graphs"]
    base, gbase = x["off"][x["inst"]], gr["noff"][gr["einst"]]
    return dict(kind=kind, parent=_i32(torch.where(x["parent"] < 0, x["parent"], x["parent"] - base)),
                off=_i32(x["off"]), max_n=int(x["tn"].max()), inst=_i32(x["inst"]), u=_i32(x["u"] - base),
                v=_i32(x["v"] - base), edges=_i32(gr["edges"] - gbase[:, None]), eoff=_i32(gr["eoff"]),
                noff=_i32(gr["noff"]), total_n=int(gr["noff"][-1]))


# ------------------------------------------------------------------ one pass


def run(state):
    kind = state["kind"]
    if kind == "tree":
        h = etl.lca_preprocess(state["parent"], workspace=state["ws"])
        out = dict(lca=h.query(state["u"], state["v"]))
        if state["arrays"]:
            out.update(h.arrays())
        return out
    if kind == "query":
        return state["handle"].query(state["u"], state["v"])
    if kind == "inlabel":
        h = etl.lca_preprocess(state["parent"], methods=("inlabel",))
        return h.query_inlabel(state["u"], state["v"])
    if kind == "list_rank":
        return etl.list_rank(state["succ"], state["head"])
    if kind == "bridges":
        return etl.find_bridges(state["edges"], state["n"])
    h = etl.lca_preprocess_batch(state["parent"], state["off"], state["max_n"])
    lca = h.query_batch(state["inst"], state["u"], state["v"])
    mask = etl.find_bridges_batch(state["edges"], state["eoff"], state["noff"], state["total_n"])
    return dict(lca=lca, bridges=mask)


def work(case):
    """Parent 4 B a node, a query 8 B in and 4 B out (+ 4 B for its tree in a batch), the tour arrays
    16 B a node; a list 4 B in and 4 B out an element; an edge 8 B in and 1 B out. Integer work only."""
    kind = case["kind"]
    if kind in ("tree", "query", "inlabel"):
        b = 12 * case["q"]
        if kind != "query":
            b += 4 * case["n"]
        if case.get("arrays"):
            b += 16 * case["n"]
    elif kind == "list_rank":
        b = 8 * case["n"]
    elif kind == "bridges":
        b = 9 * case["m"]
    else:  # expected sizes of the log-uniform draws
        tn = (2**18 - 2**6) / math.log(2**12)
        gn = (2**16 - 2**6) / math.log(2**10)
        b = int(case["trees"] * tn * 20 + case["graphs"] * gn * 36)
    return {"bytes": b, "flops": 0}


# ------------------------------------------------------------------ the results by other means


def _jumps(parent):
    """Pointer-doubling tables of a forest: jump[k][v] = the 2^k-th ancestor of v, or n (a sentinel)."""
    n = parent.numel()
    p = torch.full((n + 1,), n, dtype=torch.long, device=DEV)
    p[:-1] = torch.where(parent < 0, torch.full_like(parent, n), parent)
    tables = [p]
    while bool((tables[-1] < n).any()):
        tables.append(tables[-1][tables[-1]])
    return tables


def _path_sums(tables, w):
    """Sum of w over each node's ancestors, itself included."""
    s = torch.cat([w, torch.zeros(1, dtype=torch.long, device=DEV)])
    for t in tables:
        s = s + s[t] * (t < w.numel())
    return s[:-1]


def _subtree_sums(tables, w):
    """Sum of w over each node's subtree (mod 2^64)."""
    s = torch.cat([w, torch.zeros(1, dtype=torch.long, device=DEV)])
    for t in tables:
        s = s.index_add(0, t, s)
        s[-1] = 0
    return s[:-1]


def _lca(tables, depth, u, v):
    a, b = torch.where(depth[u] >= depth[v], u, v), torch.where(depth[u] >= depth[v], v, u)
    up = depth[a] - depth[b]
    for k, t in enumerate(tables):
        a = torch.where((up >> k) & 1 == 1, t[a], a)
    for t in reversed(tables):
        ta, tb = t[a], t[b]
        a, b = torch.where(ta != tb, ta, a), torch.where(ta != tb, tb, b)
    return torch.where(a == b, a, tables[0][a])


def _exact_bridges(gr):
    """A tree edge is a bridge iff no extra edge leaves the subtree below it: give every extra edge a
    random key, +key at one end and -key at the other; a subtree's sum is 0 iff none leaves it (but
    for a chance of 2^-60)."""
    g = _gen(12345)
    key = torch.randint(1, 1 << 62, (gr["edges"].shape[0],), generator=g, device=DEV)
    key = torch.where(gr["child"] < 0, key, torch.zeros_like(key))
    w = torch.zeros_like(gr["parent"])
    w.index_add_(0, gr["edges"][:, 0].contiguous(), key)
    w.index_add_(0, gr["edges"][:, 1].contiguous(), -key)
    s = _subtree_sums(_jumps(gr["parent"]), w)
    c = gr["child"]
    return ((c >= 0) & (s[torch.clamp(c, min=0)] == 0)).to(torch.uint8)


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "list_rank":
        rank = torch.empty_like(x["order"])
        rank[x["order"]] = torch.arange(case["n"], device=DEV)
        return _i32(rank)
    if kind == "bridges":
        return _exact_bridges(x)
    parent = x["parent"]
    n = parent.numel()
    tables = _jumps(parent)
    depth = _path_sums(tables, torch.ones_like(parent)) - 1
    lca = _lca(tables, depth, x["u"], x["v"])
    if kind in ("query", "inlabel"):
        return _i32(lca)
    if kind == "batch":
        return dict(lca=_i32(lca - x["off"][x["inst"]]), bridges=_exact_bridges(x["graphs"]))
    out = dict(lca=_i32(lca))
    if case["arrays"]:
        size = _subtree_sums(tables, torch.ones_like(parent))
        by = torch.argsort(parent, stable=True)  # children grouped by parent, in ascending label order
        before = torch.cumsum(size[by], 0) - size[by]
        p = parent[by]
        first = torch.ones_like(p, dtype=torch.bool)
        first[1:] = p[1:] != p[:-1]
        start = before[torch.cummax(torch.where(first, torch.arange(n, device=DEV), torch.zeros_like(p)), 0)[0]]
        step = torch.empty_like(parent)
        step[by] = torch.where(p < 0, torch.zeros_like(p), 1 + before - start)
        pre = _path_sums(tables, step)
        order = torch.empty_like(pre)
        order[pre] = torch.arange(n, device=DEV)
        out.update(pre=_i32(pre), depth=_i32(depth), size=_i32(size), order=_i32(order))
    return out
