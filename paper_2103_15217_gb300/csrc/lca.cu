// Lowest common ancestors by RMQ over the Euler tour (Sec. 3.1), for a tree
// given as a parent array (the input format of Sec. 3.2), or for a batch of
// independent trees preprocessed and queried together.
//
// Preprocessing (all on one stream, no host synchronisation):
//   1. link_children (sort.cu): first child and next sibling of every node, children in ascending
//      label order (the grouping step of Sec. 2.1), and validation (for a batch, also local parent
//      ids turned into global ones: node v of instance i has global id node_off[i] + v).
//   2. k_link_roots chains the tours of a batch, root i's closing bracket -> root i+1's opening
//      bracket, so one list covers all trees.
//   3. k_tour_assemble: the Euler tour's list in bracket form. Node v owns two list elements, 2v (the
//      arc entering v from its parent, an opening bracket) and 2v+1 (the arc leaving v, a closing
//      bracket). succ(2v) = 2*firstchild(v) or 2v+1; succ(2c+1) = 2*nextsibling(c) or 2*parent(c)+1.
//      This is succ(e) = next(twin(e)) of Sec. 2.1 with the cyclic list cut at the root: the root's
//      two brackets start and end its tour. Leaves are contracted on the way.
//   4. list ranking (rank.cu), counting opening brackets on the way.
//   5. k_node_stats: preorder = opening brackets before 2v; depth =
//      2*pre - rank(2v) (opening minus closing brackets before it, the +1/-1
//      prefix sum of Sec. 2); size = (rank(2v+1) - rank(2v) + 1) / 2. In a
//      chained batch, tree i occupies preorder positions node_off[i] ..
//      node_off[i+1]-1 and depth / size come out per tree.
//   6. k_parent_pre: Q[i] = pre(parent(order[i])), level 0 of the range-minimum table, in preorder, with
//      the in-block prefix / suffix minima of the blocked table.
//   7. the rest of the range-minimum table over Q (rmq.cu): by default the sparse table over blocks of
//      32 (the blocked two-level table), else a full sparse table; sized for the largest tree.
//
// Query: for u != v with i = min(pre u, pre v), j = max(...), every node with
// preorder in (i, j] is a proper descendant of LCA(u, v), and the child of the
// LCA on the path to the later end lies in that range; so the minimum of Q
// over (i, j] is pre(LCA). This is the depth-minimum of the RMQ reduction
// (the node of least depth in the range is a child of the LCA) with the
// answer read directly: one min, no argmin and no tie-breaking.
#include <climits>
#include <type_traits>

#include "etl_internal.cuh"

namespace etl {
namespace {

__device__ __forceinline__ int64_t gtid() { return blockIdx.x * int64_t(blockDim.x) + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return int64_t(gridDim.x) * blockDim.x; }

// node_off must be 0 = off[0] < off[1] < ... < off[k] = total (every instance non-empty)
__global__ void k_check_offsets(const int32_t *__restrict__ off, int32_t k, int32_t total,
                                int32_t *__restrict__ bad, int32_t *__restrict__ status) {
    pdl_prologue();
    for (int64_t i = gtid(); i < k; i += gstride()) {
        const int32_t b = off[i], e = off[i + 1];
        if (b < 0 || e > total || b >= e || (i == 0 && b != 0) || (i == k - 1 && e != total)) {
            set_status(status, ETL_EINVAL);
            *bad = 1;
        }
    }
}

// everything a build starts from: no children, cleared counters and status, the batch's offsets
__global__ void k_lca_init(int32_t n, int32_t *__restrict__ head, int64_t zeros, int32_t *__restrict__ zero,
                           int32_t *__restrict__ status) {
    pdl_prologue();
    if (gtid() == 0) *status = 0;
    for (int64_t i = gtid(); i < n; i += gstride()) head[i] = -1;
    for (int64_t i = gtid(); i < zeros; i += gstride()) zero[i] = 0;
}

// One store per node. A leaf v's brackets are adjacent in the tour: 2v jumps straight to the successor of
// 2v+1 with weight 2 (top bit set), and 2v+1 is off the list. Roots are never contracted. All accesses
// are coalesced (the closing brackets' successors were scattered to random places before, which made
// this step 0.26 ms for 2^24 nodes; now 0.07).
template <class S>  // void: successors
__global__ void k_tour_assemble(const int32_t *__restrict__ par, const int32_t *__restrict__ head,
                                const int32_t *__restrict__ next, int32_t n, const int32_t *__restrict__ roots,
                                const int32_t *__restrict__ root_of, int32_t *__restrict__ list_head,
                                void *__restrict__ list, int32_t *__restrict__ status) {
    pdl_prologue();
    if (roots && gtid() == 0) {  // one tree; k_link_roots does it for a batch
        *list_head = 2 * *root_of;
        if (*roots != 1) set_status(status, ETL_EBADTREE);
    }
    for (int64_t t = gtid(); t < n; t += gstride()) {
        const int32_t p = __ldcs(par + t), h = __ldcs(head + t), x = __ldcs(next + t);
        // leave t -> enter next sibling, or leave p; leave a root -> enter the next root
        const int32_t c = x >= 0 ? 2 * x : p >= 0 ? 2 * p + 1 : x < -1 ? 2 * (-2 - x) : ETL_END;
        const bool one = h < 0 && p >= 0;                                 // a leaf, and no root
        const int32_t a = one ? int32_t(uint32_t(c) | 0x80000000u) : h >= 0 ? 2 * h : 2 * int32_t(t) + 1;
        if constexpr (std::is_same<S, Slot8>::value)
            static_cast<ulonglong2 *>(list)[t] = make_ulonglong2(S::make(a), one ? S::off_list() : S::make(c));
        else if constexpr (std::is_same<S, Slot4d>::value)
            static_cast<uint2 *>(list)[t] = make_uint2(S::make(a), one ? S::off_list() : S::make(c));
        else
            static_cast<int2 *>(list)[t] = make_int2(a, one ? ETL_END : c);
    }
}

// exactly one root per instance; leave root i -> enter root i+1 (or end of the list after the last
// tree); the list starts at the first root's opening bracket
__global__ void k_link_roots(const int32_t *__restrict__ root_cnt, const int32_t *__restrict__ root_of, int32_t k,
                             int32_t n, int32_t *__restrict__ next, int32_t *__restrict__ list_head,
                             int32_t *__restrict__ status) {
    pdl_prologue();
    if (gtid() == 0) *list_head = 2 * root_of[0];
    for (int64_t i = gtid(); i < k; i += gstride()) {
        if (root_cnt[i] != 1) set_status(status, ETL_EBADTREE);
        const int32_t r = root_of[i];
        if (r < 0 || r >= n) continue;
        const int32_t nr = (i + 1 < k) ? root_of[i + 1] : -1;
        next[r] = (nr >= 0 && nr < n) ? -2 - nr : -1;  // told apart from a sibling by its sign
    }
}

// The two records of a node, side by side
struct NodeRecs {
    int32_t sa, sb;       // sublists of the opening and closing bracket
    int32_t ra, rb, oa;   // their offsets, and the opening brackets before the first one, in the sublists
    bool ok, leaf;        // both on the list; contracted: the closing bracket is ranked right after
};
__device__ __forceinline__ NodeRecs node_recs(ulonglong2 q) {
    NodeRecs r;
    r.leaf = Slot8::leaf(q.x) || Slot8::off(q.y);
    r.ok = !Slot8::raw(q.x) && !Slot8::off(q.x) && (r.leaf || !Slot8::raw(q.y));
    r.sa = Slot8::sid(q.x, 0);
    r.sb = r.leaf ? r.sa : Slot8::sid(q.y, 0);
    r.ra = int32_t(Slot8::lr(q.x, 0));
    r.rb = int32_t(Slot8::lr(q.y, 0));
    r.oa = int32_t(Slot8::lo(q.x));
    return r;
}
__device__ __forceinline__ NodeRecs node_recs(uint2 q) {
    NodeRecs r;
    r.leaf = Slot4d::off(q.y);
    r.ok = !Slot4d::raw(q.x) && !Slot4d::off(q.x) && (r.leaf || !Slot4d::raw(q.y));
    r.sa = Slot4d::sid(q.x, 0);
    r.sb = r.leaf ? r.sa : Slot4d::sid(q.y, 0);
    r.ra = int32_t(Slot4d::lr(q.x, 0));
    r.rb = int32_t(Slot4d::lr(q.y, 0));
    r.oa = int32_t(Slot4d::lo(q.x, uint32_t(r.ra)));
    return r;
}

// next (null: plain node ids): order[] entries carry what k_parent_pre needs to know of the node in their
// top bits, 0: it has children, 1: a leaf with a next sibling, 2: a leaf without. kIlp nodes per thread and
// step (2^24 nodes: two 268 us, one 275, four 312).
template <class Q, int kIlp>
__global__ void k_node_stats(RankResult rr, int32_t n, const int32_t *__restrict__ next, int32_t *__restrict__ pre,
                             int32_t *__restrict__ depth, int32_t *__restrict__ size, int32_t *__restrict__ order,
                             int32_t *__restrict__ status) {
    pdl_prologue();
    const Q *recs = static_cast<const Q *>(rr.recs);
    for (int64_t base = blockIdx.x * int64_t(blockDim.x) * kIlp + threadIdx.x; base < n; base += gstride() * kIlp) {
        NodeRecs r[kIlp];
        int2 A[kIlp];
        int32_t rb[kIlp];
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int64_t t = base + int64_t(j) * blockDim.x;
            r[j].ok = false;
            if (t < n) r[j] = node_recs(__ldcs(recs + t));
            r[j].ok = r[j].ok && r[j].sa >= 0 && r[j].sa < rr.rcap && r[j].sb >= 0 && r[j].sb < rr.rcap;
        }
#pragma unroll
        for (int j = 0; j < kIlp; ++j)
            if (r[j].ok) {
                A[j] = __ldg(rr.first2 + r[j].sa);
                rb[j] = r[j].leaf ? 0 : __ldg(&rr.first2[r[j].sb].x);
            }
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int64_t t = base + int64_t(j) * blockDim.x;
            if (t >= n) continue;
            if (!r[j].ok) {
                set_status(status, ETL_EBADTREE);  // not on the list from the root: malformed input
                pre[t] = depth[t] = size[t] = -1;
                continue;
            }
            const int32_t r0 = A[j].x + r[j].ra, r1 = r[j].leaf ? r0 + 1 : rb[j] + r[j].rb;
            const int32_t p = A[j].y + r[j].oa, sz = (r1 - r0 + 1) >> 1;
            __stcs(pre + t, p);
            __stcs(depth + t, 2 * p - r0);
            __stcs(size + t, sz);
            uint32_t kind = 0;
            if (next) {
                const int32_t x = __ldcs(next + t);
                kind = sz > 1 ? 0u : x >= 0 ? 1u : 2u;
            }
            if (p >= 0 && p < n) order[p] = int32_t(uint32_t(t) | kind << 30);
        }
    }
}

constexpr int32_t kFewNodes = 1 << 21;
constexpr int32_t kRecsHere = 1 << 20;

// Q in preorder: position i holds pre(parent(order[i])). If the node before i has children, it is i's
// parent: Q[i] = i - 1. If it is a leaf with a next sibling, i is that sibling: Q[i] = Q[i - 1]. Only after
// a leaf that is a last child (the rest: 30% of a random tree's positions, none of a path's) parent[] and
// pre[] have to be read at random places. A warp takes a block of 32 positions, kIlp blocks at a time, and
// leaves the block's prefix / suffix minima and its result, too (table: x, (pm, sm) pairs, top row 0 of the
// blocked layout; BLOCKED false: x only). RECS: the nodes' query records (below) instead of the pairs, in
// random order: up to kRecsHere nodes, whose records fit L2 well, that beats a launch of its own that
// gathers the pairs (whole preprocessing and n / 4 queries, us: 2^16 nodes 78.2 -> 76.9, 2^20 193.6 -> 189.1,
// 2^21 293.8 -> 302.2, 2^24 1775 -> 2380). tagged = order as k_node_stats left it, order = without tags.
// 2^24 nodes: random 153 us, path 72, with two gathers per position and a pass of its own for the
// blocks 307 and 379.
template <bool BLOCKED, bool RECS, int kIlp>
__global__ void __launch_bounds__(256)
    k_parent_pre(const int32_t *__restrict__ parent, const int32_t *__restrict__ pre,
                 const int32_t *__restrict__ tagged, int32_t n, int64_t nblk, int32_t *__restrict__ order,
                 int32_t *__restrict__ table, int4 *__restrict__ nrec, const int32_t *__restrict__ root_of,
                 const int32_t *__restrict__ size, int32_t *__restrict__ status) {
    pdl_prologue();
    if (root_of && gtid() == 0) {  // a single tree's root opens its tour and spans the tree
        const int32_t r = *root_of;
        if (r < 0 || r >= n || pre[r] != 0 || size[r] != n) set_status(status, ETL_EBADTREE);
    }
    const int64_t N = nblk * kRmqBlock, warps = gstride() / kWarp, warp = gtid() / kWarp;
    const int lane = threadIdx.x & 31;
    int32_t *top = table + 3 * N;
    for (int64_t b0 = warp * kIlp; b0 < nblk; b0 += warps * kIlp) {
        int32_t w[kIlp], before[kIlp], q[kIlp], sz[kIlp];
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int64_t i = (b0 + j) * kRmqBlock + lane;
            w[j] = b0 + j < nblk && i < n ? __ldg(tagged + i) : -1;
            before[j] = lane == 0 && b0 + j < nblk && i > 0 ? __ldg(tagged + i - 1) : -1;
        }
        if (RECS) {
#pragma unroll
            for (int j = 0; j < kIlp; ++j) {
                const int32_t v = w[j] & 0x3fffffff;
                sz[j] = v < n ? __ldg(size + v) : 0;
            }
        }
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int32_t up = __shfl_up_sync(kFull, w[j], 1);
            if (lane) before[j] = up;
            uint32_t kind = uint32_t(before[j]) >> 30;  // 3: no node before
            if (lane == 0 && kind == 1) kind = 2;       // the sibling's Q is another warp's
            before[j] = int32_t(kind);
            q[j] = -1;
            const int64_t i = (b0 + j) * kRmqBlock + lane;
            if (kind == 0) {
                q[j] = int32_t(i - 1);
            } else if (kind >= 2 && b0 + j < nblk && i < n) {
                const int32_t v = w[j] & 0x3fffffff;
                q[j] = v < n ? __ldg(parent + v) : -1;
            }
        }
#pragma unroll
        for (int j = 0; j < kIlp; ++j)
            if (before[j] >= 2) q[j] = (q[j] >= 0 && q[j] < n) ? __ldg(pre + q[j]) : -1;  // a root's is never asked for
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            if (b0 + j >= nblk) break;
            const int64_t i = (b0 + j) * kRmqBlock + lane;
            const unsigned known = __ballot_sync(kFull, before[j] != 1) & (lanemask_lt() | (1u << lane));
            int32_t x = __shfl_sync(kFull, q[j], 31 - __clz(known));  // lane 0 is always known
            if (i < n) {
                __stcs(order + i, w[j] & 0x3fffffff);
                __stcs(table + i, x);
            } else if (BLOCKED) {
                x = INT_MAX;
                table[i] = x;
            }
            if (BLOCKED) {
                int32_t a = x, c = x;
#pragma unroll
                for (int d = 1; d < kRmqBlock; d <<= 1) {
                    const int32_t ua = __shfl_up_sync(kFull, a, d), dc = __shfl_down_sync(kFull, c, d);
                    if (lane >= d) a = min(a, ua);
                    if (lane + d < kRmqBlock) c = min(c, dc);
                }
                if (!RECS)
                    __stcs(reinterpret_cast<int2 *>(table + N) + i, make_int2(a, c));
                else if (i < n && (w[j] & 0x3fffffff) < n)
                    nrec[w[j] & 0x3fffffff] = make_int4(int32_t(i), a, c, sz[j]);
                if (lane == kRmqBlock - 1) top[b0 + j] = a;
            }
        }
    }
}

// root i must open its tree at preorder off[i] and span the whole instance
__global__ void k_check_instances(const int32_t *__restrict__ root_of, const int32_t *__restrict__ off, int32_t k,
                                  int32_t n, const int32_t *__restrict__ pre, const int32_t *__restrict__ size,
                                  int32_t *__restrict__ status) {
    pdl_prologue();
    for (int64_t i = gtid(); i < k; i += gstride()) {
        const int32_t b = off ? off[i] : 0, e = off ? off[i + 1] : n;
        const int32_t r = root_of[i];
        if (r < 0 || r >= n || pre[r] != b || size[r] != e - b) set_status(status, ETL_EBADTREE);
    }
}

struct LcaView {
    int32_t n, k, levels;
    int64_t ld;
    const int32_t *pre, *order, *table, *hstatus, *off;
    BlockedView<OpMin> bv;  // the blocked table (when built instead of the full one)
    int64_t max_len;        // longest range the table answers
    const int4 *nrec;       // blocked table: per node (pre, pm[pre], sm[pre], size)
};

// Per node w with p = pre(w): the per-position entries of the blocked table that a query can need
// from w's side, pm[p] (w has the larger preorder number) and sm[p] (the smaller one), with p and
// size(w), so that a query reads two 16-byte records instead of pre[] twice, then pm and sm. The
// table stores (pm, sm) pairs, so this is one 8-byte gather per node.
template <int kIlp>  // nodes per thread per step, their gathers in flight together
__global__ void k_node_rec(const int32_t *__restrict__ pre, const int32_t *__restrict__ size,
                           const int2 *__restrict__ pmsm, int32_t n, int4 *__restrict__ nrec) {
    pdl_prologue();
    const int64_t step = gstride() * kIlp;
    for (int64_t base = blockIdx.x * int64_t(blockDim.x) * kIlp + threadIdx.x; base < n; base += step) {
        int32_t p[kIlp];
        int2 e[kIlp];
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int64_t w = base + int64_t(j) * blockDim.x;
            p[j] = w < n ? __ldcs(pre + w) : -1;
            e[j] = (p[j] >= 0 && p[j] < n) ? __ldg(pmsm + p[j]) : make_int2(INT_MAX, INT_MAX);  // bad tree: flagged
        }
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int64_t w = base + int64_t(j) * blockDim.x;
            if (w < n) __stcs(nrec + w, make_int4(p[j], e[j].x, e[j].y, __ldcs(size + w)));
        }
    }
}

// Queries per thread and step. Up to kQueryFew the memory behind them fits L2 or they are too few to fill
// the GPU four to a thread: 2^20 queries of a 2^22-node tree 22.1 us with four, 19.1 with one, 2^14 5.4 and
// 2.5; 2^22 69 and 69; 2^24 queries of a 2^24-node tree, bound by DRAM, 564 and 583.
constexpr int kQueryIlp = 4;
constexpr int64_t kQueryFew = int64_t(1) << 22;

// min of x[lo..hi], a range inside one block of the blocked table (at most 32 entries, one line)
__device__ __forceinline__ int32_t inblock_min(const int32_t *__restrict__ x, int32_t lo, int32_t hi) {
    int32_t m = __ldg(x + lo);
    for (int32_t j = lo + 1; j <= hi; ++j) m = min(m, __ldg(x + j));
    return m;
}

// Each thread answers ILP queries at once so that their dependent gathers
// (pre, table, order) overlap in flight. BATCH: ids are local to the
// instance inst[i] and so is the answer.
template <bool BATCH, bool BLOCKED, int ILP>
__global__ void __launch_bounds__(256)
    k_lca_query(LcaView h, const int32_t *__restrict__ inst, const int32_t *__restrict__ u,
                const int32_t *__restrict__ v, int64_t q, int32_t *__restrict__ out, int32_t *__restrict__ status) {
    pdl_prologue();
    const bool bad_tree = *h.hstatus != 0;
    const int64_t stride = gstride();
    for (int64_t base = gtid(); base < q; base += stride * ILP) {
        int32_t a[ILP], b[ILP], lo[ILP], hi[ILP], res[ILP], ofs[ILP];
        bool need[ILP], ok[ILP];
#pragma unroll
        for (int k = 0; k < ILP; ++k) {
            const int64_t i = base + k * stride;
            need[k] = false;
            ok[k] = false;
            res[k] = -1;
            ofs[k] = 0;
            a[k] = b[k] = 0;
            if (i < q) {
                a[k] = __ldcs(u + i);
                b[k] = __ldcs(v + i);
                int32_t lim = h.n;
                if (BATCH) {
                    const int32_t t = __ldcs(inst + i);
                    if (t >= 0 && t < h.k) {
                        ofs[k] = __ldg(h.off + t);
                        lim = __ldg(h.off + t + 1) - ofs[k];
                    } else {
                        lim = 0;
                    }
                }
                ok[k] = a[k] >= 0 && a[k] < lim && b[k] >= 0 && b[k] < lim;
                if (!ok[k]) set_status(status, ETL_EBADQUERY);
            }
        }
#pragma unroll
        for (int k = 0; k < ILP; ++k) {
            if (!ok[k] || bad_tree) continue;
            if (a[k] == b[k]) {
                res[k] = a[k];
            } else if (BLOCKED) {
                const int4 ra = __ldg(h.nrec + ofs[k] + a[k]), rb = __ldg(h.nrec + ofs[k] + b[k]);
                const bool a_first = ra.x < rb.x;
                const int4 x = a_first ? ra : rb, y = a_first ? rb : ra;  // x earlier in preorder
                lo[k] = x.x + 1;
                hi[k] = y.x;
                need[k] = hi[k] - lo[k] + 1 <= h.max_len;  // cannot fail unless max_n was understated
                if (!need[k]) {
                    set_status(status, ETL_EINVAL);
                } else if (y.x < x.x + x.w) {  // y lies in x's subtree: x is the answer
                    need[k] = false;
                    res[k] = a_first ? a[k] : b[k];
                } else if ((x.x >> kRmqBlockLog2) != (hi[k] >> kRmqBlockLog2)) {
                    // across blocks: x is no ancestor of y, so Q at pre(x) (x's parent, the LCA or below
                    // it) cannot lower the minimum and the range may start at pre(x) itself: sm[pre x]
                    // and pm[pre y] come with the records, whole blocks between from the top table
                    int32_t m = min(x.z, y.y);
                    const int32_t bl = (x.x >> kRmqBlockLog2) + 1, bh = (hi[k] >> kRmqBlockLog2) - 1;
                    if (bl <= bh) {
                        const int l = 31 - __clz(bh - bl + 1);
                        const int32_t *row = h.bv.top + int64_t(l) * h.bv.nblk;
                        m = min(m, min(__ldg(row + bl), __ldg(row + bh - (1 << l) + 1)));
                    }
                    lo[k] = m;
                    hi[k] = -1;  // answered
                }
            } else {
                const int32_t pa = __ldg(h.pre + ofs[k] + a[k]), pb = __ldg(h.pre + ofs[k] + b[k]);
                lo[k] = min(pa, pb) + 1;
                hi[k] = max(pa, pb);
                need[k] = hi[k] - lo[k] + 1 <= h.max_len;  // cannot fail unless max_n was understated
                if (!need[k]) set_status(status, ETL_EINVAL);
            }
        }
#pragma unroll
        for (int k = 0; k < ILP; ++k)
            if (need[k] && hi[k] >= 0)  // in one block (blocked table), or the full table
                lo[k] = BLOCKED ? inblock_min(h.bv.x, lo[k], hi[k]) : sparse_query<false>(h.table, h.ld, lo[k], hi[k]);
#pragma unroll
        for (int k = 0; k < ILP; ++k) {
            const int64_t i = base + k * stride;
            if (i >= q) continue;
            if (need[k]) res[k] = __ldg(h.order + lo[k]) - ofs[k];
            __stcs(out + i, res[k]);
        }
    }
}

int grid_for(int64_t work, int threads) {
    int64_t blocks = ceil_div(work, threads);
    const int64_t cap = int64_t(num_sms()) * (2048 / threads) * 4;
    if (blocks > cap) blocks = cap;
    return int(blocks < 1 ? 1 : blocks);
}

void free_handle(etl_lca_s *h) {
    if (!h) return;
    if (h->arena) {  // the device arrays belong to the caller's workspace
        delete h;
        return;
    }
    cudaStream_t s = h->stream;
    for (void *p : {h->block, h->inrec, h->inpath, h->tour_table, static_cast<void *>(h->tpos)})
        if (p) cudaFreeAsync(p, s);
    delete h;
}

// n nodes in k >= 1 trees; node_off (device, k+1 entries) is null for one tree
etl_status lca_build(const int32_t *parent, int32_t n, const int32_t *node_off, int32_t k, int32_t max_n,
                     bool with_table, cudaStream_t s, etl_lca_t *out) {
    const bool batch = node_off != nullptr;
    etl_lca_s *h = new etl_lca_s;
    h->arena = current_arena() != nullptr;
    h->n = n;
    h->k = k;
    h->stream = s;
    h->levels = max_n > 1 ? sparse_levels(max_n - 1) : 1;
    h->has_table = with_table;
    h->ld = sparse_ld(n);
    h->blocked = rmq_params().blocked;
    h->bl = blocked_layout(n, max_n);
    const size_t table_bytes = (h->blocked ? size_t(h->bl.elems()) : size_t(h->ld) * size_t(h->levels)) * 4;
    // one allocation for all arrays of the handle, each 256-byte aligned in it
    const size_t nb = size_t(n) * sizeof(int32_t);
    const size_t bytes[8] = {nb, nb, nb, nb, sizeof(int32_t), with_table ? table_bytes : 0,
                             with_table && h->blocked ? size_t(n) * sizeof(int4) : 0,
                             batch ? size_t(k + 1) * sizeof(int32_t) : 0};
    size_t at[8], total = 0;
    for (int i = 0; i < 8; ++i) {
        at[i] = total;
        total += (bytes[i] + 255) & ~size_t(255);
    }
    if (dev_alloc(&h->block, total, s) != cudaSuccess) {
        h->block = nullptr;
        free_handle(h);
        return ETL_ENOMEM;
    }
    auto part = [&](int i) { return bytes[i] ? reinterpret_cast<int32_t *>(static_cast<char *>(h->block) + at[i]) : nullptr; };
    h->pre = part(0);
    h->depth = part(1);
    h->size = part(2);
    h->order = part(3);
    h->status = part(4);
    h->table = part(5);
    h->nrec = part(6);
    h->node_off = part(7);
    if (!batch && n <= kTinyNodes && (h->blocked || !with_table)) {
        const etl_status st = build_tiny_tree(parent, h, s);
        if (st) {
            free_handle(h);
            return st;
        }
        *out = h;
        return ETL_OK;
    }
    if (batch) copy_d2d_async(h->node_off, node_off, size_t(k + 1) * sizeof(int32_t), s);
    etl_status st = ETL_OK;
    {
        Workspace ws(s);
        const RankForm form = rank_form(2 * int64_t(n), true);
        const bool recs_here = h->blocked && n <= kRecsHere;
        const bool few = n <= kFewNodes;  // one node per thread and step fills the GPU better
        void *list = form == RankForm::kSlots8 ? static_cast<void *>(ws.get<ulonglong2>(n)) : ws.get<int2>(n);  // 2n elements
        int32_t *head = ws.get<int32_t>(n), *next = ws.get<int32_t>(n);
        // cleared: offsets invalid, the ranking's counter, roots per tree, a root of each, link_children's words
        const int64_t zeros = 2 + 2 * int64_t(k) + link_words(n);
        int32_t *zero = ws.get<int32_t>(zeros + 1), *list_head = zero + zeros;
        int32_t *bad = zero, *rank_zero = zero + 1, *root_cnt = zero + 2, *root_of = root_cnt + k, *words = root_of + k;
        int32_t *gparent = batch ? ws.get<int32_t>(n) : nullptr;
        if (!ws.ok()) st = ETL_ENOMEM;
        const int32_t *par = batch ? gparent : parent;
        if (!st) {
            {
                PhaseTimer pt("lca.init", s);
                launch(k_lca_init, grid_for(n, 256), 256, 0, s, n, head, zeros, zero, h->status);
                note_launch();
                if (batch) {
                    launch(k_check_offsets, grid_for(k, 256), 256, 0, s, h->node_off, k, n, bad, h->status);
                    note_launch();
                }
            }
            st = link_children(parent, n, h->node_off, k, bad, gparent, head, next, root_cnt, root_of, words, h->status,
                               ws);
        }
        if (!st) {
            PhaseTimer pt("lca.succ", s);
            if (batch) {
                launch(k_link_roots, grid_for(k, 256), 256, 0, s, root_cnt, root_of, k, n, next, list_head, h->status);
                note_launch();
            }
            launch(form == RankForm::kSlots8   ? k_tour_assemble<Slot8>
                   : form == RankForm::kSlots4 ? k_tour_assemble<Slot4d>
                                               : k_tour_assemble<void>,
                   grid_for(n, 256), 256, 0, s, par, head, next, n, batch ? nullptr : root_cnt, root_of, list_head, list,
                   h->status);
            note_launch();
            st = last_launch();
        }
        int32_t *tagged = head;  // order[] with tags; the first children are not needed once the list is built
        RankResult rr{};
        if (!st) st = list_rank(list, 2 * int64_t(n), list_head, 0, true, 2 * int64_t(n), rank_zero, h->status, ws, &rr);
        if (!st) {
            PhaseTimer pt("lca.node_stats", s);
            launch(rr.wide ? (few ? k_node_stats<ulonglong2, 1> : k_node_stats<ulonglong2, 2>) : k_node_stats<uint2, 2>,
                   grid_for(n, 256), 256, 0, s, rr, n,
                   with_table ? next : nullptr, h->pre, h->depth, h->size, with_table ? tagged : h->order, h->status);
            note_launch();
            if (batch || !with_table) {  // k_parent_pre looks at a single tree's root
                launch(k_check_instances, grid_for(k, 256), 256, 0, s, root_of, batch ? h->node_off : nullptr, k, n,
                       h->pre, h->size, h->status);
                note_launch();
            }
            st = last_launch();
        }
        if (!st && with_table) {
            PhaseTimer pt("lca.parent_pre", s);
            launch(!h->blocked ? k_parent_pre<false, false, 4>
                   : recs_here ? k_parent_pre<true, true, 1>
                   : few       ? k_parent_pre<true, false, 1>
                               : k_parent_pre<true, false, 4>,
                   grid_for(n, few ? 256 : 256 * 4), 256, 0, s, par, h->pre, tagged, n, h->bl.nblk, h->order, h->table,
                   static_cast<int4 *>(h->nrec), batch ? nullptr : root_of, h->size, h->status);
            note_launch();
            st = last_launch();
        }
        if (!st && with_table)
            st = h->blocked ? blocked_top<OpMin>(h->table + 3 * h->bl.nblk * kRmqBlock, h->bl, s)
                            : sparse_table_build<false>(h->table, n, h->levels, s);
        if (!st && with_table && h->blocked && !recs_here) {
            PhaseTimer pt("lca.node_rec", s);
            launch(few ? k_node_rec<1> : k_node_rec<4>, grid_for(n, 256), 256, 0, s, h->pre, h->size,
                   reinterpret_cast<const int2 *>(h->table + h->bl.nblk * kRmqBlock), n, static_cast<int4 *>(h->nrec));
            note_launch();
            st = last_launch();
        }
    }
    if (st) {
        free_handle(h);
        return st;
    }
    *out = h;
    return ETL_OK;
}

etl_status query_launch(etl_lca_t h, const int32_t *inst, const int32_t *u, const int32_t *v, int64_t q,
                        int32_t *out, int32_t *status, cudaStream_t s) {
    LcaView view{h->n,     h->k,      h->levels, h->ld,
                 h->pre,   h->order,  h->table,  h->status,
                 h->node_off, blocked_view<OpMin>(h->table, h->bl),
                 h->blocked ? blocked_max_len(h->bl) : (int64_t(1) << h->levels) - 1,
                 static_cast<const int4 *>(h->nrec)};
    PhaseTimer pt("lca.query", s);
    const bool few = q <= kQueryFew;
    const int grid = grid_for(few ? q : ceil_div(q, kQueryIlp), 256);
    auto kernel = h->blocked ? (inst ? (few ? k_lca_query<true, true, 1> : k_lca_query<true, true, kQueryIlp>)
                                     : (few ? k_lca_query<false, true, 1> : k_lca_query<false, true, kQueryIlp>))
                             : (inst ? (few ? k_lca_query<true, false, 1> : k_lca_query<true, false, kQueryIlp>)
                                     : (few ? k_lca_query<false, false, 1> : k_lca_query<false, false, kQueryIlp>));
    launch(kernel, grid, 256, 0, s, view, inst, u, v, q, out, status);
    note_launch();
    return last_launch();
}

}  // namespace
}  // namespace etl

using namespace etl;

extern "C" etl_status lca_preprocess(const int32_t *parent, int32_t n, void *stream, etl_lca_t *out) {
    if (!out) return ETL_EINVAL;
    *out = nullptr;
    if (!parent || n < 1 || n > (1 << 30) - 1) return ETL_EINVAL;
    return lca_build(parent, n, nullptr, 1, n, true, static_cast<cudaStream_t>(stream), out);
}

etl_status lca_build_inlabel_impl(etl_lca_t h, const int32_t *parent, cudaStream_t s);
etl_status lca_build_tour_impl(etl_lca_t h, const int32_t *parent, cudaStream_t s);

extern "C" etl_status lca_preprocess_ex(const int32_t *parent, int32_t n, int32_t flags, void *stream,
                                        etl_lca_t *out) {
    if (!out) return ETL_EINVAL;
    *out = nullptr;
    constexpr int32_t kAll = ETL_LCA_RMQ | ETL_LCA_INLABEL | ETL_LCA_TOUR_RMQ;
    if (!parent || n < 1 || n > (1 << 30) - 1 || !(flags & kAll) || (flags & ~kAll)) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    etl_status st = lca_build(parent, n, nullptr, 1, n, (flags & ETL_LCA_RMQ) != 0, s, out);
    if (!st && (flags & ETL_LCA_INLABEL)) st = lca_build_inlabel_impl(*out, parent, s);
    if (!st && (flags & ETL_LCA_TOUR_RMQ)) st = lca_build_tour_impl(*out, parent, s);
    if (st && *out) {
        free_handle(*out);
        *out = nullptr;
    }
    return st;
}

extern "C" etl_status lca_preprocess_batch(const int32_t *parent, const int32_t *node_off, int32_t k,
                                           int32_t total_n, int32_t max_n, void *stream, etl_lca_t *out) {
    if (!out) return ETL_EINVAL;
    *out = nullptr;
    if (!parent || !node_off || k < 1 || total_n < k || total_n > (1 << 30) - 1 || max_n < 1 || max_n > total_n)
        return ETL_EINVAL;
    return lca_build(parent, total_n, node_off, k, max_n, true, static_cast<cudaStream_t>(stream), out);
}

extern "C" etl_status lca_query(etl_lca_t h, const int32_t *u, const int32_t *v, int64_t q, int32_t *out,
                                int32_t *status, void *stream) {
    if (!h || h->node_off || !h->has_table || q < 0 || q > (int64_t(1) << 40)) return ETL_EINVAL;
    if (q == 0) return ETL_OK;
    if (!u || !v || !out) return ETL_EINVAL;
    return query_launch(h, nullptr, u, v, q, out, status, static_cast<cudaStream_t>(stream));
}

extern "C" etl_status lca_query_batch(etl_lca_t h, const int32_t *inst, const int32_t *u, const int32_t *v,
                                      int64_t q, int32_t *out, int32_t *status, void *stream) {
    if (!h || !h->node_off || q < 0 || q > (int64_t(1) << 40)) return ETL_EINVAL;
    if (q == 0) return ETL_OK;
    if (!inst || !u || !v || !out) return ETL_EINVAL;
    return query_launch(h, inst, u, v, q, out, status, static_cast<cudaStream_t>(stream));
}

extern "C" etl_status lca_status(etl_lca_t h, int32_t *status) {
    if (!h || !status) return ETL_EINVAL;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return ETL_ECUDA;
    if (cudaMemcpy(status, h->status, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess) return ETL_ECUDA;
    return ETL_OK;
}

extern "C" etl_status lca_arrays(etl_lca_t h, const int32_t **pre, const int32_t **depth, const int32_t **size,
                                 const int32_t **order) {
    if (!h) return ETL_EINVAL;
    if (pre) *pre = h->pre;
    if (depth) *depth = h->depth;
    if (size) *size = h->size;
    if (order) *order = h->order;
    return ETL_OK;
}

extern "C" etl_status lca_export(etl_lca_t h, int32_t *pre, int32_t *depth, int32_t *size, int32_t *order,
                                 void *stream) {
    if (!h) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t nb = size_t(h->n) * sizeof(int32_t);
    int32_t *dst[4] = {pre, depth, size, order};
    const int32_t *src[4] = {h->pre, h->depth, h->size, h->order};
    for (int i = 0; i < 4; ++i)
        if (dst[i] && copy_d2d_async(dst[i], src[i], nb, s) != cudaSuccess) return ETL_ECUDA;
    return ETL_OK;
}

extern "C" etl_status lca_free(etl_lca_t h) {
    if (!h) return ETL_OK;
    free_handle(h);
    return cudaGetLastError() == cudaSuccess ? ETL_OK : ETL_ECUDA;
}
