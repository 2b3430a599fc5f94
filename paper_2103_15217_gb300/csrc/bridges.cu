// Bridges by the Tarjan-Vishkin method (Sec. 4.1) on one GPU.
//
// Phase 1, spanning forest: a lock-free hook-and-compress connected-components
//   pass in the style the paper takes from Jaiganesh and Burtscher: every edge
//   finds the roots of its two ends (with path halving) and hooks the one of
//   lower priority under the other with a CAS. A CAS that succeeds joins two
//   different trees, so its edge is a forest edge; exactly n - c succeed.
//   The successful edges are appended to the forest's list as they are found.
// Phase 2, Euler tour of the forest (Sec. 2.1): forest edge t owns half-edges
//   2t = (u_t, v_t) and 2t+1 = (v_t, u_t), so twin(a) = a ^ 1. Every half-edge
//   is pushed onto its tail's list (one exchange; the order inside a vertex's
//   group is free, any cyclic order gives an Euler tour); next(a) is the entry
//   after it, cyclically; succ(a) = next(twin(a)). Each component's cyclic list
//   is cut in front of the first half-edge of its root, and the component
//   lists are chained into one list in any order, which is ranked once
//   (rank.cu). Tour position = rank + 1; position 0 stands before the tour.
// Phase 3, low / high: with tin(x) = position of the half-edge entering x (a
//   root gets the position just before its component), the subtree of u is the
//   tour interval [tin(u), tout(u)], tout(u) = position of the half-edge
//   leaving u. Position p starts with (low, high) = (p, p); every non-forest
//   edge (x, w) updates the entries at tin(x) and tin(w) by atomic min / max
//   (the paper uses a segmented reduction); low(u) / high(u) are range-min /
//   -max queries over [tin(u), tout(u)]: one blocked table of (L, H) pairs by
//   default, else two full sparse tables (rmq.cu). (An entry (p, p) at a
//   position p inside the interval, also where no vertex is entered, cannot
//   take the minimum below tin(u) or the maximum above tout(u).)
// Phase 4, the test: forest edge {u, parent(u)} is a bridge iff
//   low(u) >= tin(u) and high(u) <= tout(u), i.e. no non-forest edge leaves
//   the subtree of u. (Sec. 4.1 states the condition the other way round;
//   low or high escaping the subtree's interval is the NON-bridge case,
//   since such an edge reconnects the subtree with the rest of the graph.)
#include <climits>

#include "etl_internal.cuh"

namespace etl {
namespace {

constexpr int64_t kFindCap = int64_t(1) << 26;  // bound on pointer-chasing steps of one edge

// forest: [0] edges found, [1] first half-edge of the component list (the ranked list's head), [2] zero
__global__ void k_init(int32_t n, int32_t *__restrict__ par, int32_t *__restrict__ head, int32_t *__restrict__ tin,
                       int32_t *__restrict__ forest) {
    pdl_prologue();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        forest[0] = 0;
        forest[1] = ETL_END;
        forest[2] = 0;
    }
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x) {
        par[v] = int32_t(v);
        head[v] = -1;
        tin[v] = 0;
    }
}

// both ends of edge e; one 8-byte load if the caller's array allows it
__device__ __forceinline__ int2 load_edge(const int32_t *__restrict__ edges, int64_t e, bool aligned) {
    return aligned ? __ldcs(reinterpret_cast<const int2 *>(edges) + e)
                   : make_int2(__ldcs(edges + 2 * e), __ldcs(edges + 2 * e + 1));
}
inline bool edges_aligned(const int32_t *edges) { return (reinterpret_cast<uintptr_t>(edges) & 7) == 0; }

// Root of x with path halving; -1 if the step budget runs out. MIN (only where ancestors have smaller ids):
// pointers never move down again, whatever order the writes of several lanes come in.
template <bool MIN>
__device__ __forceinline__ int32_t find_root(int32_t *par, int32_t x, int64_t &budget) {
    while (budget-- > 0) {
        const int32_t p = __ldcg(par + x);
        if (p == x) return p;
        const int32_t gp = __ldcg(par + p);
        if (gp == p) return p;
        if (MIN)
            atomicMin(par + x, gp);
        else
            atomicExch(par + x, gp);  // only non-roots are rewritten, always to an ancestor
        x = gp;
    }
    return -1;
}

// The edges are cut into chunks of kHookChunk consecutive edges; one launch hooks positions c0 .. c1 - 1
// of the chunk sequence, kHookIlp positions per block step. With `spread` (batches of graphs) the
// chunks are grouped into superchunks of kHookSuper that are visited in a permuted order
// (superchunk s of the sequence is s * P mod nsuper, P = 2^31 - 1, a prime above any superchunk
// count, so the map is a bijection), the chunks of a superchunk in order. The blocks running at one
// time then work on ~150 regions of 64 KB of edges spread over the whole list: in a batch of many
// small graphs, a contiguous sweep puts thousands of threads on one graph's few roots, where their
// CAS attempts collide and retry (measured: 11.4 -> 4 ms on 2048 graphs), and a first slice of the
// sequence samples every graph of the batch, not the first ones only. A single graph keeps the
// contiguous order, which measured faster on it (0.7 against 1.3 ms on 2^25 shuffled edges).
constexpr int kHookChunk = 256;
constexpr int kHookIlp = 4;
// All edges go in one launch while their number is at most 700 sqrt(vertices), else a first slice, a compression
// and the rest. One launch saves two others and the walk over all vertices between them; with more edges the
// walks that meet no compressed path cost more. Hook launches of random graphs, us, in one and in slices, and
// where the two are equal: 1025 vertices, 16 edges each 17 and 25, 32 32 and 30, equal at some 25000 edges; 4097,
// 8 20 and 27, 16 29 and 28, 60000; 16385, 4 20 and 30, 8 29 and 31, 136000; 32769, 4 28 and 32, 8 54 and 36,
// 160000; 65537, 2 24 and 35, 4 50 and 37, 180000; 92682, 2 31 and 37, 4 67 and 38, 250000. The line stays
// below; hard graphs (long paths) gain from one launch at all of these sizes (16385, 4 each 20 and 34).
// Half as many edges again in the first slice up to kHookMoreFirst vertices: 4 edges each on 2^15.3 vertices 42
// -> 33, 2^17 63 -> 45 (hard 51 -> 49), 2^18 67 -> 63 (68 -> 65), 2^19 89 -> 92, 2^20 122 -> 144 (132 -> 134);
// there the slice itself is the dearer part.
inline bool hook_at_once(int64_t n, int64_t m) { return m * m <= 490000 * n; }
constexpr int32_t kHookMoreFirst = 1 << 18;
constexpr int kHookSuper = 32;

// number of positions of the chunk sequence over m edges (whole superchunks)
inline int64_t hook_positions(int64_t m) {
    return ceil_div(ceil_div(m, kHookChunk), kHookSuper) * kHookSuper;
}

__device__ __forceinline__ int64_t hook_chunk(int64_t c, int64_t nsuper, bool spread) {
    constexpr int64_t kP = 2147483647;
    return spread ? ((c / kHookSuper) * kP % nsuper) * kHookSuper + c % kHookSuper : c;
}

// Roots are hooked under roots of higher priority. Priorities are a strict total order, so the forest stays
// acyclic. The root named by *giant (if any: the most frequent root after a compression, i.e. the giant
// component's) ranks above all, so it never moves: once the giant component has formed, every later hook
// leaves the paths of its members as they are (with a fixed order its root moves whenever a higher one joins,
// and every member's path grows by a step). The others are ordered by a mixed id (MurmurHash3's 32-bit
// finalizer, a bijection), or, where the component's label is to be its smallest vertex (BY_ID), by the id.
// By ids a path whose vertices are numbered along it is hooked into one chain, and an edge that comes late
// climbs it alone, 0.5 us for two steps. Whole calls, us, by ids and now: paths in order of 2^17 vertices 1170
// to 6690 and 89, of 2^20 31700 and 254 (from their end 27700 and 257), a cycle of 2^14 4120 and 58, a path of
// 2^14, where no edge comes late, 48 and 58. On the easy graph of 2^22 vertices, whose labels are permuted, 1420
// and 1428 (by ids the popular parents lie side by side), on the hard one 1222 and 1184.
template <bool BY_ID>
__device__ __forceinline__ uint32_t hook_key(int32_t v) {
    uint32_t h = uint32_t(v);
    if (BY_ID) return h;
    h = (h ^ (h >> 16)) * 0x85ebca6bu;
    h = (h ^ (h >> 13)) * 0xc2b2ae35u;
    return h ^ (h >> 16);
}
template <bool BY_ID>
__device__ __forceinline__ bool hook_above(int32_t a, int32_t b, int32_t giant) {  // a ranks above b
    return a == giant || (b != giant && hook_key<BY_ID>(a) < hook_key<BY_ID>(b));
}

// Most edges join two vertices that already point at the same node; those cost two loads, all of a
// block step's in flight together. The others go to a queue in shared memory, and the block hooks them
// 256 at a time with every lane busy (one lane's walk to a root held up the other 31 before). A lane walks
// up from both ends of its edge at once, halving both paths, until they meet (usually well below the root)
// or both end at roots. Halving is done by exchanges: a plain store to a sector that others read takes over
// 1 us. A node's pointer is read from L2, its parent's through L1: parents are few and popular (reads of
// one address are served one after another by its L2 slice). A stale one does no harm: it still leads to
// an ancestor, what is no root any more makes the CAS fail, and the walk goes on from its own pointer. The
// edges that join two trees are appended to the forest's list, one counter update per round. Easy graph of
// 2^22 vertices and 2^25 edges, whole pass: 735 us without the queue, 680 with it, 530 with the giant root
// known to the walks, 500 with exchanges, 478 with both walks at once (hard graph 557 -> 470, 512 graphs
// 588 -> 456); the two loads per edge of its 31.4M later edges alone take 210 us.
// skip (may be null): edges to leave out; is_tree (may be null): 1 for edges whose hook succeeded, and
// then is_bridge is cleared and forest_count, tuv (both ends of forest edge t) and tedge (its edge) are written too
template <bool BY_ID>
__global__ void __launch_bounds__(kHookChunk)
    k_hook(const int32_t *__restrict__ edges, bool aligned, int64_t m, int64_t c0, int64_t c1, int ilp, bool spread,
           int32_t n, int32_t *__restrict__ par, uint8_t *__restrict__ is_tree, uint8_t *__restrict__ is_bridge,
           const uint8_t *__restrict__ skip, const int32_t *__restrict__ d_giant, int32_t *__restrict__ forest_count, int2 *__restrict__ tuv,
           int32_t *__restrict__ tedge, int32_t *__restrict__ status) {
    pdl_prologue();
    __shared__ int32_t qa[kHookChunk * (kHookIlp + 1)], qb[kHookChunk * (kHookIlp + 1)], qe[kHookChunk * (kHookIlp + 1)];
    __shared__ int queued, wins[kHookChunk / 32], first;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t giant = d_giant ? *d_giant : 0;  // vertex 0 ranks above all by its id, and by its key
    const int64_t nsuper = ((m + kHookChunk - 1) / kHookChunk + kHookSuper - 1) / kHookSuper;
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
    const int64_t step = int64_t(gridDim.x) * ilp;
    for (int64_t c = c0 + int64_t(blockIdx.x) * ilp; c < c1; c += step) {
        int2 ab[kHookIlp];
        int64_t e[kHookIlp];
        bool ok[kHookIlp];
        int32_t pa[kHookIlp], pb[kHookIlp];
#pragma unroll
        for (int j = 0; j < kHookIlp; ++j) {
            e[j] = j < ilp && c + j < c1 ? hook_chunk(c + j, nsuper, spread) * kHookChunk + threadIdx.x : m;
            ok[j] = e[j] < m;
            if (ok[j]) ab[j] = load_edge(edges, e[j], aligned);
        }
#pragma unroll
        for (int j = 0; j < kHookIlp; ++j) {
            if (!ok[j]) continue;
            if (is_tree) is_tree[e[j]] = is_bridge[e[j]] = 0;
            if (skip && skip[e[j]]) {
                ok[j] = false;
            } else if (ab[j].x < 0 || ab[j].x >= n || ab[j].y < 0 || ab[j].y >= n) {
                set_status(status, ETL_EBADGRAPH);
                ok[j] = false;
            } else {
                pa[j] = __ldcg(par + ab[j].x);
                pb[j] = __ldcg(par + ab[j].y);
            }
        }
#pragma unroll
        for (int j = 0; j < kHookIlp; ++j)
            if (ok[j] && pa[j] != pb[j]) {
                const int i = atomicAdd(&queued, 1);
                qa[i] = ab[j].x;
                qb[i] = ab[j].y;
                qe[i] = int32_t(e[j]);
            }
        __syncthreads();
        const int have = queued, keep = c + step < c1 ? have & (kHookChunk - 1) : 0;  // full rounds, all in the end
        for (int i0 = keep; i0 < have; i0 += kHookChunk) {
            const int i = i0 + threadIdx.x;
            bool won = false;
            if (i < have) {
                int32_t a = qa[i], b = qb[i];
                int64_t budget = kFindCap;
                while (true) {  // both walks at once, up to a node on both
                    if (budget-- <= 0) {
                        set_status(status, ETL_ETIMEOUT);
                        break;
                    }
                    const int32_t pa = a == giant ? a : __ldcg(par + a), pb = b == giant ? b : __ldcg(par + b);
                    if (pa == pb) break;
                    const bool ta = pa == a || pa == giant, tb = pb == b || pb == giant;
                    const int32_t ga = ta ? pa : __ldca(par + pa);
                    const int32_t gb = tb ? pb : __ldca(par + pb);
                    if (ga != pa) atomicExch(par + a, ga);  // only non-roots are rewritten, always to an ancestor
                    if (gb != pb) atomicExch(par + b, gb);
                    if (ga == gb) break;
                    a = ga;
                    b = gb;
                    if ((ga != pa && ga != giant) || (gb != pb && gb != giant)) continue;
                    const bool a_up = hook_above<BY_ID>(a, b, giant);
                    const int32_t hi = a_up ? b : a, lo = a_up ? a : b;  // hi goes under lo
                    if (atomicCAS(par + hi, hi, lo) == hi) {
                        won = true;
                        break;
                    }  // someone hooked one of the roots meanwhile: on from them
                }
            }
            if (!is_tree) continue;
            const unsigned ball = __ballot_sync(kFull, won);
            if (lane == 0) wins[warp] = __popc(ball);
            __syncthreads();
            int before = __popc(ball & lanemask_lt()), total = 0;
            for (int w = 0; w < kHookChunk / 32; ++w) {
                if (w < warp) before += wins[w];
                total += wins[w];
            }
            if (threadIdx.x == 0 && total) first = atomicAdd(forest_count, total);
            __syncthreads();
            if (won) {
                const int64_t t = int64_t(first) + before;
                is_tree[qe[i]] = 1;
                tuv[t] = make_int2(qa[i], qb[i]);
                tedge[t] = qe[i];
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) queued = keep;
        __syncthreads();
    }
}

// The root most often reached from kGiantSample vertices spread over [0, n): the giant component's when
// there is one. k_hook takes it for a root, so every walk goes on to a true one. One block
constexpr int kGiantSample = 1024;

__device__ void sample_giant(const int32_t *__restrict__ par, int32_t n, int32_t *__restrict__ giant) {
    constexpr int kSlots = 2 * kGiantSample;  // open-addressing table of (root, count)
    __shared__ int32_t key[kSlots], cnt[kSlots];
    __shared__ unsigned long long best;
    for (int j = threadIdx.x; j < kSlots; j += blockDim.x) {
        key[j] = -1;
        cnt[j] = 0;
    }
    if (threadIdx.x == 0) best = 0;
    __syncthreads();
    for (int i0 = threadIdx.x; i0 < kGiantSample; i0 += 4 * blockDim.x) {
        int32_t r[4], p[4];
        int64_t budget = kFindCap;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r[j] = int32_t((uint64_t(i0 + j * int(blockDim.x)) * 2654435761u + 12345u) % uint64_t(n));
        bool more = true;
        while (more && budget-- > 0) {
            more = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = __ldcg(par + r[j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                more |= p[j] != r[j];
                r[j] = p[j];
            }
        }
        for (int j = 0; j < 4; ++j) {
            if (i0 + j * int(blockDim.x) >= kGiantSample) break;
            uint32_t h = (uint32_t(r[j]) * 2654435761u) >> 21;  // 11 bits: kSlots = 2048
            for (int probe = 0; probe < kSlots; ++probe, h = (h + 1) & (kSlots - 1)) {
                const int32_t prev = atomicCAS(&key[h], -1, r[j]);
                if (prev == -1 || prev == r[j]) {
                    atomicAdd(&cnt[h], 1);
                    break;
                }
            }
        }
    }
    __syncthreads();
    // largest count, then smallest root id: pack (count, ~root) and take the maximum
    for (int j = threadIdx.x; j < kSlots; j += blockDim.x)
        if (cnt[j]) atomicMax(&best, (static_cast<unsigned long long>(cnt[j]) << 32) | uint32_t(~uint32_t(key[j])));
    __syncthreads();
    if (threadIdx.x == 0) *giant = int32_t(~uint32_t(best & 0xffffffffu));
}

// Up to kGiantBeside vertices the giant is found by an extra block of the compression (2^14 vertices 36 ->
// 31 us for both hook launches), beyond by a launch after it, when its walks are one step: the table in
// shared memory takes L1 from all blocks of the compression and of what runs next (hard graph of 2^22
// vertices 518 us against 470).
constexpr int32_t kGiantBeside = 1 << 18;

// Points every vertex at its root. EXACT: at the root itself in the end (the labels of components hooked in
// id order); otherwise a lane that halves a path late may leave a vertex at an inner node, and the last
// block finds the giant root meanwhile
template <bool EXACT, bool GIANT>
__global__ void k_compress(int32_t n, int32_t *__restrict__ par, int32_t *__restrict__ giant, int32_t *__restrict__ status) {
    pdl_prologue();
    int64_t blocks = gridDim.x;
    if (GIANT) {
        --blocks;
        if (blockIdx.x == blocks) {
            sample_giant(par, n, giant);
            return;
        }
    }
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n; v += blocks * blockDim.x) {
        int64_t budget = kFindCap;
        const int32_t p = __ldcg(par + v), r = find_root<EXACT>(par, p, budget);
        if (r < 0) {
            set_status(status, ETL_ETIMEOUT);
        } else if (r != p) {
            if (EXACT)
                atomicMin(par + v, r);
            else
                atomicExch(par + v, r);
        }
    }
}

__global__ void k_giant(const int32_t *__restrict__ par, int32_t n, int32_t *__restrict__ giant) {
    pdl_prologue();
    sample_giant(par, n, giant);
}

// next[a] = the half-edge pushed onto its tail's list before a (-1: none). Half-edges of one tail in a
// warp are linked by the warp and pushed as one run.
__global__ void k_link_arcs(const int32_t *__restrict__ tuv, const int32_t *__restrict__ forest,
                            int32_t *__restrict__ head, int32_t *__restrict__ next) {
    pdl_prologue();
    const int64_t len = 2 * int64_t(*forest);
    const int lane = threadIdx.x & 31;
    for (int64_t base = blockIdx.x * int64_t(blockDim.x); base < len; base += int64_t(gridDim.x) * blockDim.x) {
        const int64_t a = base + threadIdx.x;
        const int32_t x = a < len ? tuv[a] : -1;
        const unsigned peers = __match_any_sync(kFull, x >= 0 ? x : -1 - lane);
        const int first = __ffs(peers) - 1;
        int32_t old = -1;
        if (x >= 0 && lane == first) old = atomicExch(head + x, int32_t(a));
        old = __shfl_sync(kFull, old, first);
        const unsigned above = lane < 31 ? peers >> (lane + 1) : 0u;
        if (a < len) next[a] = above ? int32_t(a) + __ffs(above) : old;
    }
}

// What follows the twin of half-edge a (tail x): the next half-edge of x. The last one is followed by the
// first, but at a component's root, where the list is cut: there by the first half-edge of the component
// chained before. on: lanes with a half-edge (all lanes call)
__device__ __forceinline__ int32_t arc_after(int32_t a, int32_t nb, bool on, const int32_t *__restrict__ tuv,
                                             const int32_t *__restrict__ par, const int32_t *__restrict__ head,
                                             int32_t *__restrict__ chain) {
    bool cut = false;
    if (on && nb < 0) {
        const int32_t x = tuv[a];
        nb = head[x];
        cut = par[x] == x;
    }
    const unsigned m = __ballot_sync(kFull, cut);
    if (m) {  // the warp's roots form one run of the component list
        const int lane = threadIdx.x & 31, first = __ffs(m) - 1;
        const unsigned above = lane < 31 ? m >> (lane + 1) : 0u;
        const int32_t after = __shfl_sync(kFull, nb, above ? lane + __ffs(above) : lane);
        int32_t old = ETL_END;
        if (lane == first) old = atomicExch(chain, nb);
        old = __shfl_sync(kFull, old, first);
        if (cut) nb = above ? after : old;
    }
    return nb;
}

// the list's elements (len of them, half-edges beyond the forest off it), twins side by side
template <class S>
__global__ void k_forest_list(const int32_t *__restrict__ tuv, int32_t *__restrict__ forest,
                              const int32_t *__restrict__ par, const int32_t *__restrict__ head,
                              const int32_t *__restrict__ next, int64_t len, typename S::T *__restrict__ list) {
    pdl_prologue();
    const int64_t T = forest[0], pairs = (len + 1) / 2;
    for (int64_t base = blockIdx.x * int64_t(blockDim.x); base < pairs; base += int64_t(gridDim.x) * blockDim.x) {
        const int64_t t = base + threadIdx.x;
        const bool on = t < T;
        const int2 nb = on ? __ldcs(reinterpret_cast<const int2 *>(next) + t) : make_int2(0, 0);
        const int32_t s1 = arc_after(int32_t(2 * t), nb.x, on, tuv, par, head, forest + 1);
        const int32_t s0 = arc_after(int32_t(2 * t + 1), nb.y, on, tuv, par, head, forest + 1);
        if (2 * t < len) list[2 * t] = on ? S::make(s0) : S::off_list();
        if (2 * t + 1 < len) list[2 * t + 1] = on ? S::make(s1) : S::off_list();
    }
}

// tour positions of forest edges: the half-edge ranked first goes down into the child; and of roots
__global__ void k_forest_tin(RankResult rr, const int32_t *__restrict__ forest, int32_t n, const int2 *__restrict__ tuv,
                             const int32_t *__restrict__ par, const int32_t *__restrict__ head,
                             int32_t *__restrict__ tin, int32_t *__restrict__ child, int32_t *__restrict__ etin,
                             int32_t *__restrict__ etout) {
    pdl_prologue();
    const int64_t T = *forest;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < n; t += int64_t(gridDim.x) * blockDim.x) {
        const int32_t h = par[t] == t ? head[t] : -1;
        if (h >= 0) tin[t] = ~rank_at(rr, h);  // a root's, just before its first half-edge, is marked by its sign
        if (t >= T) continue;
        const int32_t r0 = rank_at(rr, 2 * t), r1 = rank_at(rr, 2 * t + 1);
        if (r0 < 0 || r1 < 0) {  // cannot happen for a forest built above; keep memory safe
            if (child) child[t] = 0;
            etin[t] = etout[t] = -1;
            continue;
        }
        const int2 uv = tuv[t];
        const int32_t c = r0 < r1 ? uv.y : uv.x;
        const int32_t a = min(r0, r1) + 1, b = max(r0, r1) + 1;
        tin[c] = a;
        if (child) child[t] = c;
        etin[t] = a;
        etout[t] = b;
    }
}

// low / high of position p are L[p << shift], H[p << shift]
__global__ void k_lowhigh_init(int64_t P, int32_t *__restrict__ L, int32_t *__restrict__ H, int shift) {
    pdl_prologue();
    for (int64_t p = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; p < P; p += int64_t(gridDim.x) * blockDim.x)
        L[p << shift] = H[p << shift] = int32_t(p);
}

// Updates of one position are served one after another. With many edges per position most of them change
// nothing, which a load shows (CHECK), through L1: an entry that is out of date there only lets an update pass.
// Random graphs, whole calls without and with the check, us: 10 vertices and 655361 edges 434 and 98, 100 and
// 4.2M 1737 and 314, 1000 and 1.0M 226 and 201, 256001 98 and 103, 64001 61 and 64, 10000 and 2.6M (128 per
// position) 160 and 144, 320001 88 and 90, 100000 and 25.6M 692 and 631.
constexpr int64_t kCheckEach = 128, kCheckEdges = 1 << 19;  // edges per position, edges

template <bool CHECK>
__global__ void k_nontree_minmax(const int32_t *__restrict__ edges, bool aligned, int64_t m, int32_t n,
                                 const uint8_t *__restrict__ is_tree, const int32_t *__restrict__ tin, int64_t P,
                                 int32_t *L, int32_t *H, int shift) {
    pdl_prologue();
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < m; e += int64_t(gridDim.x) * blockDim.x) {
        if (__ldcs(is_tree + e)) continue;
        const int2 ab = load_edge(edges, e, aligned);
        const int32_t a = ab.x, b = ab.y;
        if (a < 0 || a >= n || b < 0 || b >= n || a == b) continue;
        int32_t ta = __ldg(tin + a), tb = __ldg(tin + b);
        const bool root = ta < 0 || tb < 0;  // then it is the earlier end
        if (ta < 0) ta = ~ta;
        if (tb < 0) tb = ~tb;
        const int64_t lo = min(ta, tb), hi = max(ta, tb);
        if (hi >= P || lo == hi) continue;
        // of the four updates only the one lowering the later end's low and the one raising the earlier
        // end's high can change anything; a root's entry is in no interval of its component (its position
        // is the last one of another component's)
        if (!root && !(CHECK && __ldca(H + (lo << shift)) >= hi)) atomicMax(H + (lo << shift), int32_t(hi));
        if (!(CHECK && __ldca(L + (hi << shift)) <= lo)) atomicMin(L + (hi << shift), int32_t(lo));
    }
}

// bridges among the forest edges; the mask is zero before, and stays so on a data error
__global__ void k_bridge_test2(const int32_t *__restrict__ forest, const int32_t *__restrict__ etin,
                               const int32_t *__restrict__ etout, BlockedView<OpMinMax> lh, int64_t P,
                               const int32_t *__restrict__ tedge, const int32_t *__restrict__ status,
                               uint8_t *__restrict__ is_bridge) {
    pdl_prologue();
    const int64_t T = *status == 0 ? *forest : 0;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < T; t += int64_t(gridDim.x) * blockDim.x) {
        const int32_t a = etin[t], b = etout[t];
        if (a < 0 || b >= P || a >= b) continue;
        const int2 own = __ldg(lh.x + a);  // the child's own edges alone mostly show that it is none
        if (own.x < a || own.y > b) continue;
        const int2 r = blocked_query<OpMinMax>(lh, a, b);  // (low, high) of the subtree
        if (r.x >= a && r.y <= b) is_bridge[tedge[t]] = 1;
    }
}

__global__ void k_bridge_test(const int32_t *__restrict__ forest, const int32_t *__restrict__ etin,
                              const int32_t *__restrict__ etout, const int32_t *__restrict__ Lt,
                              const int32_t *__restrict__ Ht, int64_t P, int64_t ld, const int32_t *__restrict__ tedge,
                              const int32_t *__restrict__ status, uint8_t *__restrict__ is_bridge) {
    pdl_prologue();
    const int64_t T = *status == 0 ? *forest : 0;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < T; t += int64_t(gridDim.x) * blockDim.x) {
        const int32_t a = etin[t], b = etout[t];
        if (a < 0 || b >= P || a >= b) continue;
        const int32_t low = sparse_query<false>(Lt, ld, a, b);
        const int32_t high = sparse_query<true>(Ht, ld, a, b);
        if (low >= a && high <= b) is_bridge[tedge[t]] = 1;
    }
}

}  // namespace

CcParams &cc_params() {
    static CcParams p;
    return p;
}

namespace {

int grid_for(int64_t work, int threads) {
    int64_t blocks = ceil_div(work, threads);
    const int64_t cap = int64_t(num_sms()) * (2048 / threads) * 4;
    if (blocks > cap) blocks = cap;
    return int(blocks < 1 ? 1 : blocks);
}

// chunks per block step: as many as leave every resident block a step; and the grid
int hook_ilp(int64_t chunks) {
    const int64_t each = chunks / (int64_t(num_sms()) * (2048 / kHookChunk));
    return int(each < 1 ? 1 : each < kHookIlp ? each : kHookIlp);
}
int hook_grid(int64_t chunks) {
    const int64_t blocks = ceil_div(chunks, hook_ilp(chunks)), most = int64_t(num_sms()) * (2048 / kHookChunk);
    return int(blocks < most ? (blocks < 1 ? 1 : blocks) : most);
}

// ---- the hybrid of Sec. 4.3: parents and levels of the rooted forest from its Euler tour, then
// Chaitanya-Kothapalli marking: every non-tree edge walks both ends up to their LCA and marks the
// tree edges on the way (a tree edge is named by its child); unmarked tree edges are bridges

__global__ void k_tour_pm(const int32_t *__restrict__ forest, const int32_t *__restrict__ etin,
                          const int32_t *__restrict__ etout, int64_t P, int32_t *__restrict__ val) {
    pdl_prologue();
    const int64_t T = *forest;
    if (blockIdx.x == 0 && threadIdx.x == 0) val[0] = 0;  // the virtual head
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < T; t += int64_t(gridDim.x) * blockDim.x) {
        const int32_t a = etin[t], b = etout[t];
        if (a < 0 || b >= P || a >= b) continue;
        val[a] = 1;   // down into the child: one level deeper
        val[b] = -1;  // back up
    }
}

__global__ void k_tree_records(int32_t n, const int32_t *__restrict__ forest, const int32_t *__restrict__ tuv,
                               const int32_t *__restrict__ child, const int32_t *__restrict__ etin,
                               const int32_t *__restrict__ excl, int64_t P, int2 *__restrict__ trec,
                               uint8_t *__restrict__ mark) {
    pdl_prologue();
    const int64_t T = *forest;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < T; t += int64_t(gridDim.x) * blockDim.x) {
        const int32_t c = child[t], a = etin[t];
        if (a < 0 || a >= P) continue;
        const int32_t p = tuv[2 * t] == c ? tuv[2 * t + 1] : tuv[2 * t];
        trec[c] = make_int2(p, excl[a + 1]);  // (parent, level): level = prefix of +-1 at the child's entry
        mark[c] = 0;
    }
}

__global__ void k_tree_records_init(int32_t n, int2 *__restrict__ trec) {
    pdl_prologue();
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x)
        trec[v] = make_int2(-1, 0);  // roots and isolated vertices
}

__global__ void k_ck_mark(const int32_t *__restrict__ edges, int64_t m, int32_t n, const uint8_t *__restrict__ is_tree,
                          const int2 *__restrict__ trec, uint8_t *__restrict__ mark, int32_t *__restrict__ status) {
    pdl_prologue();
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < m; e += int64_t(gridDim.x) * blockDim.x) {
        if (is_tree[e]) continue;
        int32_t a = edges[2 * e], b = edges[2 * e + 1];
        if (a < 0 || a >= n || b < 0 || b >= n || a == b) continue;
        int2 ra = __ldg(trec + a), rb = __ldg(trec + b);
        int64_t steps = 0;
        while (a != b) {
            if (++steps > 2 * int64_t(n)) {
                set_status(status, ETL_ETIMEOUT);
                break;
            }
            if (ra.y >= rb.y) {
                mark[a] = 1;
                a = ra.x;
                if (a < 0 || a >= n) break;
                ra = __ldg(trec + a);
            } else {
                mark[b] = 1;
                b = rb.x;
                if (b < 0 || b >= n) break;
                rb = __ldg(trec + b);
            }
        }
    }
}

__global__ void k_ck_bridges(const int32_t *__restrict__ forest, const int32_t *__restrict__ child,
                             const uint8_t *__restrict__ mark, const int32_t *__restrict__ tedge,
                             const int32_t *__restrict__ status, uint8_t *__restrict__ is_bridge) {
    pdl_prologue();
    const int64_t T = *status == 0 ? *forest : 0;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < T; t += int64_t(gridDim.x) * blockDim.x)
        if (!mark[child[t]]) is_bridge[tedge[t]] = 1;
}

etl_status hybrid_marking(const int32_t *edges, int64_t m, int32_t n, const uint8_t *is_tree, const int32_t *tuv,
                          const int32_t *tedge, const int32_t *forest, const int32_t *child, const int32_t *etin,
                          const int32_t *etout, int64_t P, uint8_t *is_bridge, int32_t *st, Workspace &ws) {
    cudaStream_t s = ws.stream();
    int32_t *val = ws.get<int32_t>(P), *excl = ws.get<int32_t>(P + 1);
    int2 *trec = ws.get<int2>(n);
    uint8_t *mark = ws.get<uint8_t>(n);
    if (!ws.ok()) return ETL_ENOMEM;
    const int gn = grid_for(n, 256);
    {
        PhaseTimer pt("hybrid.levels", s);
        launch(k_tour_pm, gn, 256, 0, s, forest, etin, etout, P, val);
        note_launch();
    }
    etl_status rc = last_launch();
    if (!rc) rc = scan_exclusive_i32(val, excl, P, ws);
    if (rc) return rc;
    PhaseTimer pt("hybrid.mark", s);
    launch(k_tree_records_init, gn, 256, 0, s, n, trec);
    note_launch();
    launch(k_tree_records, gn, 256, 0, s, n, forest, tuv, child, etin, excl, P, trec, mark);
    note_launch();
    launch(k_ck_mark, grid_for(m, 256), 256, 0, s, edges, m, n, is_tree, trec, mark, st);
    note_launch();
    launch(k_ck_bridges, gn, 256, 0, s, forest, child, mark, tedge, st, is_bridge);
    note_launch();
    return last_launch();
}

// the whole Tarjan-Vishkin pipeline on a graph with global ids; st is a zeroed device status word.
// hybrid: instead of low / high, the Chaitanya-Kothapalli marking on the same rooted forest
etl_status bridges_core(const int32_t *edges, int64_t m, int32_t n, uint8_t *is_bridge, int32_t *st,
                        Workspace &ws, bool hybrid = false, bool spread = false) {
    cudaStream_t s = ws.stream();
    const int64_t A = 2 * int64_t(n - 1);  // half-edge capacity of a spanning forest
    const int64_t N = A > 0 ? A : 1;        // elements of the ranked list
    const int64_t P = A + 1;                // tour positions 0 .. A
    const int levels = sparse_levels(P);
    const int64_t ld = sparse_ld(P);
    const bool blocked = rmq_params().blocked, aligned = edges_aligned(edges);
    const BlockedLayout bl = blocked_layout(P, P);
    int32_t *par = ws.get<int32_t>(n), *head = ws.get<int32_t>(n), *tin = ws.get<int32_t>(n);
    uint8_t *is_tree = ws.get<uint8_t>(m);
    int2 *tuv = ws.get<int2>(n);
    int32_t *arcs = reinterpret_cast<int32_t *>(tuv), *next = ws.get<int32_t>(N + 1);  // tail of / half-edge after each
    int32_t *tedge = ws.get<int32_t>(n);
    int32_t *forest = ws.get<int32_t>(3), *giant = ws.get<int32_t>(1);
    const bool wide = wide_slots(N);
    void *list = wide ? static_cast<void *>(ws.get<Slot8::T>(N)) : static_cast<void *>(ws.get<Slot4::T>(N));  // slots or successors
    int32_t *child = hybrid ? ws.get<int32_t>(n) : nullptr;
    int32_t *etin = ws.get<int32_t>(n), *etout = ws.get<int32_t>(n);
    int32_t *Lt = (hybrid || blocked) ? nullptr : ws.get<int32_t>(ld * levels);
    int32_t *Ht = (hybrid || blocked) ? nullptr : ws.get<int32_t>(ld * levels);
    int2 *LH = (!hybrid && blocked) ? ws.get<int2>(bl.elems()) : nullptr;
    if (!ws.ok()) return ETL_ENOMEM;
    etl_status rc = ETL_OK;
    const int gn = grid_for(n, 256), gm = grid_for(m, 256), gA = grid_for(N, 256);
    {
        PhaseTimer pt("br.init", s);
        launch(k_init, gn, 256, 0, s, n, par, head, tin, forest);
        note_launch();
    }
    {
        // hook a first slice of the edges, compress every path to its root, then hook the rest:
        // after the compression most finds take one step and most edges meet equal roots at once.
        // With `doubling`, the rest goes in slices that double in size, each followed by a
        // compression, so that no phase builds long paths in a fresh part of the forest.
        const CcParams &C = cc_params();
        const int64_t nchunks = hook_positions(m);
        int64_t slice = int64_t(C.first_slice_quarters) * n / 4;
        if (n <= kHookMoreFirst) slice += slice / 2;
        int64_t w = hook_at_once(n, m) ? nchunks : ceil_div(slice > 0 ? slice : 1, kHookChunk);  // chunks in the current slice
        PhaseTimer pt("br.hook", s);
        for (int64_t c0 = 0; c0 < nchunks;) {
            const int64_t c1 = (C.doubling || c0 == 0) ? (c0 + w < nchunks ? c0 + w : nchunks) : nchunks;
            if (c0 > 0) {
                const bool beside = C.giant && n <= kGiantBeside;
                if (beside)
                    launch(k_compress<false, true>, gn + 1, 256, 0, s, n, par, giant, st);
                else
                    launch(k_compress<false, false>, gn, 256, 0, s, n, par, nullptr, st);
                note_launch();
                if (C.giant && !beside) {
                    launch(k_giant, 1, kGiantSample, 0, s, par, n, giant);
                    note_launch();
                }
            }
            launch(k_hook<false>, hook_grid(c1 - c0), kHookChunk, 0, s, edges, aligned, m, c0, c1,
                   hook_ilp(c1 - c0), spread, n, par, is_tree, is_bridge, nullptr, (c0 > 0 && C.giant) ? giant : nullptr, forest,
                   tuv, tedge, st);
            note_launch();
            c0 = c1;
            w *= 2;
        }
    }
    rc = last_launch();
    if (!rc) {
        PhaseTimer pt("br.forest_list", s);
        launch(k_link_arcs, gA, 256, 0, s, arcs, forest, head, next);
        note_launch();
        if (wide)
            launch(k_forest_list<Slot8>, gA, 256, 0, s, arcs, forest, par, head, next, N, static_cast<Slot8::T *>(list));
        else
            launch(k_forest_list<Slot4>, gA, 256, 0, s, arcs, forest, par, head, next, N, static_cast<Slot4::T *>(list));
        note_launch();
        rc = last_launch();
    }
    RankResult rr{};
    if (!rc) rc = list_rank(list, N, forest + 1, 0, false, -1, forest + 2, st, ws, &rr);
    if (!rc) {
        PhaseTimer pt("br.tin", s);
        launch(k_forest_tin, gn, 256, 0, s, rr, forest, n, tuv, par, head, tin, child, etin, etout);
        note_launch();
        rc = last_launch();
    }
    if (hybrid)
        return rc ? rc : hybrid_marking(edges, m, n, is_tree, arcs, tedge, forest, child, etin, etout, P, is_bridge, st, ws);
    if (!rc) {
        PhaseTimer pt("br.lowhigh_prep", s);
        int32_t *L = blocked ? reinterpret_cast<int32_t *>(LH) : Lt, *H = blocked ? L + 1 : Ht;
        launch(k_lowhigh_init, grid_for(P, 256), 256, 0, s, P, L, H, blocked ? 1 : 0);
        note_launch();
        launch(m >= kCheckEdges && m >= kCheckEach * P ? k_nontree_minmax<true> : k_nontree_minmax<false>, gm, 256, 0, s, edges, aligned, m, n, is_tree, tin, P, L, H, blocked ? 1 : 0);
        note_launch();
        rc = last_launch();
    }
    if (blocked) {
        if (!rc) rc = blocked_build<OpMinMax>(LH, P, bl, s);
    } else {
        if (!rc) rc = sparse_table_build<false>(Lt, P, levels, s);
        if (!rc) rc = sparse_table_build<true>(Ht, P, levels, s);
    }
    if (!rc) {
        PhaseTimer pt("br.test", s);
        if (blocked)
            launch(k_bridge_test2, gn, 256, 0, s, forest, etin, etout, blocked_view<OpMinMax>(LH, bl), P, tedge, st,
                   is_bridge);
        else
            launch(k_bridge_test, gn, 256, 0, s, forest, etin, etout, Lt, Ht, P, ld, tedge, st, is_bridge);
        note_launch();
        rc = last_launch();
    }
    return rc;
}

__global__ void k_iota(int32_t n, int32_t *__restrict__ x) {
    pdl_prologue();
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x)
        x[v] = int32_t(v);
}

__global__ void k_labels_on_error(int32_t n, const int32_t *__restrict__ status, int32_t *__restrict__ label) {
    pdl_prologue();
    if (*status == 0) return;
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x)
        label[v] = -1;
}

// local edge ids of a batch -> global ids: edge e of instance i (edge_off[i] <= e < edge_off[i+1])
// joins node_off[i] + u and node_off[i] + v
__global__ void k_check_batch(const int32_t *__restrict__ eoff, const int32_t *__restrict__ noff, int32_t k,
                              int64_t m, int32_t n, int32_t *__restrict__ bad, int32_t *__restrict__ status) {
    pdl_prologue();
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < k; i += int64_t(gridDim.x) * blockDim.x) {
        const bool ok = eoff[i] >= 0 && eoff[i] <= eoff[i + 1] && eoff[i + 1] <= m && noff[i] >= 0 &&
                        noff[i] < noff[i + 1] && noff[i + 1] <= n && (i > 0 || (eoff[0] == 0 && noff[0] == 0)) &&
                        (i < k - 1 || (eoff[k] == m && noff[k] == n));
        if (!ok) {
            set_status(status, ETL_EINVAL);
            *bad = 1;
        }
    }
}

// A block takes kGlobalTile consecutive edges and looks up the instances of the first and the last, a
// thread its edge's between the two (19M edges of 512 graphs: 124 us with a search over all instances per
// edge, 67 now).
constexpr int kGlobalTile = 2048;

__global__ void __launch_bounds__(256)
    k_globalize(const int32_t *__restrict__ edges, bool aligned, int64_t m, const int32_t *__restrict__ eoff,
                const int32_t *__restrict__ noff, int32_t k, const int32_t *__restrict__ bad, int2 *__restrict__ gedges,
                int32_t *__restrict__ status) {
    pdl_prologue();
    __shared__ int32_t span[2];
    const bool unusable = *bad != 0;
    const int64_t base = int64_t(blockIdx.x) * kGlobalTile, end = min(base + kGlobalTile, m);
    if (threadIdx.x < 2 && !unusable) span[threadIdx.x] = last_at_or_before(eoff, 0, k - 1, threadIdx.x == 0 ? base : end - 1);
    __syncthreads();
    for (int64_t e = base + threadIdx.x; e < end; e += blockDim.x) {
        int2 g = make_int2(-1, -1);
        if (!unusable) {  // offsets are monotone, from 0 to m: checked before
            const int32_t i = last_at_or_before(eoff, span[0], span[1], e);
            const int32_t from = __ldg(noff + i), size = __ldg(noff + i + 1) - from;
            const int2 ab = load_edge(edges, e, aligned);
            if (ab.x >= 0 && ab.x < size && ab.y >= 0 && ab.y < size)
                g = make_int2(ab.x + from, ab.y + from);
            else
                set_status(status, ETL_EBADGRAPH);
        }
        gedges[e] = g;
    }
}

}  // namespace
}  // namespace etl

using namespace etl;

extern "C" etl_status find_bridges(const int32_t *edges, int64_t m, int32_t n, uint8_t *is_bridge, int32_t *status,
                                   void *stream) {
    if (n < 1 || n > (1 << 30) - 1 || m < 0 || m > int64_t(INT32_MAX) - 1) return ETL_EINVAL;
    if (m == 0) return ETL_OK;
    if (!edges || !is_bridge) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Workspace ws(s);
    int32_t *st = status ? status : ws.get<int32_t>(1);
    if (!ws.ok()) return ETL_ENOMEM;
    memset_async(st, 0, sizeof(int32_t), s);
    return bridges_core(edges, m, n, is_bridge, st, ws);
}

extern "C" etl_status find_bridges_batch(const int32_t *edges, const int32_t *edge_off, const int32_t *node_off,
                                         int32_t k, int64_t total_m, int32_t total_n, uint8_t *is_bridge,
                                         int32_t *status, void *stream) {
    if (k < 1 || total_n < k || total_n > (1 << 30) - 1 || total_m < 0 || total_m > int64_t(INT32_MAX) - 1)
        return ETL_EINVAL;
    if (!edge_off || !node_off) return ETL_EINVAL;
    if (total_m == 0) return ETL_OK;
    if (!edges || !is_bridge) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Workspace ws(s);
    int32_t *st = status ? status : ws.get<int32_t>(1);
    int32_t *bad = ws.get<int32_t>(1);
    int32_t *gedges = ws.get<int32_t>(2 * total_m);
    if (!ws.ok()) return ETL_ENOMEM;
    memset_async(st, 0, sizeof(int32_t), s);
    memset_async(bad, 0, sizeof(int32_t), s);
    {
        PhaseTimer pt("br.globalize", s);
        launch(k_check_batch, grid_for(k, 256), 256, 0, s, edge_off, node_off, k, total_m, total_n, bad, st);
        note_launch();
        launch(k_globalize, unsigned(ceil_div(total_m, kGlobalTile)), 256, 0, s, edges, edges_aligned(edges), total_m,
               edge_off, node_off, k, bad, reinterpret_cast<int2 *>(gedges), st);
        note_launch();
    }
    etl_status rc = last_launch();
    if (rc) return rc;
    return bridges_core(gedges, total_m, total_n, is_bridge, st, ws, false, true);
}

extern "C" etl_status two_edge_cc(const int32_t *edges, int64_t m, int32_t n, int32_t *label, int32_t *status,
                                  void *stream) {
    if (n < 1 || n > (1 << 30) - 1 || m < 0 || m > int64_t(INT32_MAX) - 1 || !label) return ETL_EINVAL;
    if (m > 0 && !edges) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Workspace ws(s);
    int32_t *st = status ? status : ws.get<int32_t>(1);
    uint8_t *is_bridge = ws.get<uint8_t>(m > 0 ? m : 1);
    if (!ws.ok()) return ETL_ENOMEM;
    memset_async(st, 0, sizeof(int32_t), s);
    etl_status rc = m > 0 ? bridges_core(edges, m, n, is_bridge, st, ws) : ETL_OK;
    if (rc) return rc;
    const int gn = grid_for(n, 256);
    PhaseTimer pt("br.two_edge_cc", s);
    launch(k_iota, gn, 256, 0, s, n, label);
    note_launch();
    if (m > 0) {  // connected components of the graph without its bridges; labels = smallest vertex
        launch(k_hook<true>, hook_grid(hook_positions(m)), kHookChunk, 0, s, edges, edges_aligned(edges), m, 0,
               hook_positions(m), hook_ilp(hook_positions(m)), false, n, label, nullptr,
               nullptr, is_bridge, nullptr, nullptr, nullptr, nullptr, st);
        note_launch();
        launch(k_compress<true, false>, gn, 256, 0, s, n, label, nullptr, st);
        note_launch();
    }
    launch(k_labels_on_error, gn, 256, 0, s, n, st, label);
    note_launch();
    return last_launch();
}

extern "C" etl_status find_bridges_hybrid(const int32_t *edges, int64_t m, int32_t n, uint8_t *is_bridge,
                                          int32_t *status, void *stream) {
    if (n < 1 || n > (1 << 30) - 1 || m < 0 || m > int64_t(INT32_MAX) - 1) return ETL_EINVAL;
    if (m == 0) return ETL_OK;
    if (!edges || !is_bridge) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Workspace ws(s);
    int32_t *st = status ? status : ws.get<int32_t>(1);
    if (!ws.ok()) return ETL_ENOMEM;
    memset_async(st, 0, sizeof(int32_t), s);
    return bridges_core(edges, m, n, is_bridge, st, ws, true);
}
