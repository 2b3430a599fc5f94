// Children of every node in ascending label order, as linked lists (the grouping step of Sec. 2.1: the
// paper sorts the arcs; a tour only needs each node's first child and next sibling).
//
//  * k_link_children pushes every node onto its parent's list, highest labels first:
//    next[c] = exchange(head[parent[c]], c). Blocks start in the order of their index, so almost every
//    list comes out ascending; only siblings whose pushes were in flight together can be swapped. The
//    lanes of a warp that share a parent are linked by the warp and pushed as one run. One random
//    exchange in an array of n words per node: 2^24 nodes in 0.13 ms, where counting the children,
//    scanning the counts and a stable 3-pass radix sort of (parent, child) pairs took 0.54 ms, and a
//    random tree's successors another 0.17 ms of random writes that the lists do not need.
//  * k_check_children finds every link that does not ascend and sorts that family's list on the spot
//    (up to kLight children, by one thread). k_sort_children takes its place on small inputs, where most do not.
//  * k_sort_heavy does longer families that are out of order: a stable LSD radix sort of their
//    (parent, child) pairs, 8 bits per pass, in one cooperative launch, which returns at once when
//    there are none (3 us). Inside a tile each warp ranks its 32-element rounds (peers with the same
//    digit by __match_any_sync or by eight ballots) with per-warp smem counters; the ranked tile is
//    staged in shared memory in digit order and written out in runs.
#include <algorithm>
#include <climits>

#include "etl_internal.cuh"

namespace etl {
namespace {

__device__ __forceinline__ int64_t gtid() { return blockIdx.x * int64_t(blockDim.x) + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return int64_t(gridDim.x) * blockDim.x; }

constexpr int kLinkThreads = 256;
constexpr int kLinkIlp = 2;  // labels per thread, from the highest down (1: 0.16 ms, 4: more siblings in flight together)
constexpr int kLight = 32;   // children of a family that one thread sorts

// Batches: blocks that run together take tiles of different parts of the list, each part from its end down, so
// that fewer siblings are pushed at one time. A part's ends cut through a tree, whose halves come in the wrong
// order, so a part holds at least 8 trees. 512 trees of 2^24 nodes in all, the check of the order: 174 us as
// one part, 136 as 8, 118 to 121 as 16 to 48, 131 as 64, 156 as 128; the pushes take the same time.
constexpr int kLinkGroups = 32;

// off / k / bad (batches): ids are local to the node's instance, gparent receives global ones. A block
// looks up the instances of its first and last label, a thread its own between the two.
template <bool BATCH>
__global__ void __launch_bounds__(kLinkThreads)
    k_link_children(const int32_t *__restrict__ parent, int32_t n, int32_t groups, const int32_t *__restrict__ off,
                    int32_t k, const int32_t *__restrict__ bad, int32_t *__restrict__ gparent, int32_t *__restrict__ head,
                    int32_t *__restrict__ next, int32_t *__restrict__ root_cnt, int32_t *__restrict__ root_of,
                    int32_t *__restrict__ status) {
    pdl_prologue();
    const bool bad_offsets = BATCH && *bad;
    int64_t tile = gridDim.x - 1 - blockIdx.x;
    if (BATCH) {
        const uint32_t each = gridDim.x / groups;
        tile = int64_t(blockIdx.x % groups) * each + (each - 1 - blockIdx.x / groups);
    }
    const int64_t top = (tile + 1) * (kLinkThreads * kLinkIlp);
    if (BATCH && tile * (kLinkThreads * kLinkIlp) >= n) return;
    __shared__ int32_t span[2];
    if (BATCH) {
        if (threadIdx.x < 2 && !bad_offsets)
            span[threadIdx.x] = last_at_or_before(
                off, 0, k - 1, threadIdx.x == 0 ? top - kLinkThreads * kLinkIlp : min(top, int64_t(n)) - 1);
        __syncthreads();
    }
    int32_t par[kLinkIlp];
#pragma unroll
    for (int j = 0; j < kLinkIlp; ++j) {
        const int64_t t = top - int64_t(j + 1) * kLinkThreads + threadIdx.x;
        par[j] = t < n ? __ldcs(parent + t) : -1;
    }
#pragma unroll
    for (int j = 0; j < kLinkIlp; ++j) {
        const int64_t t = top - int64_t(j + 1) * kLinkThreads + threadIdx.x;
        const int32_t v = int32_t(t), p = par[j];
        int32_t g = -2;
        if (t < n && !bad_offsets) {
            int32_t inst = 0, base = 0, size = n;
            if (BATCH) {
                inst = last_at_or_before(off, span[0], span[1], v);
                base = off[inst];
                size = off[inst + 1] - base;
            }
            if (p == -1) {
                atomicAdd(&root_cnt[inst], 1);
                root_of[inst] = v;
                g = -1;
            } else if (p < 0 || p >= size) {
                set_status(status, ETL_EBADTREE);
            } else {
                g = p + base;
                if (g == v) set_status(status, ETL_EBADTREE);
            }
        }
        // Where many lanes share a parent they form one run, linked in label order, which its first lane
        // pushes: pushes to one address are served one after another. The samples catch the parents with a
        // large share of the labels; matching all lanes in every warp took 15 us more for 2^24 nodes.
        const int lane = threadIdx.x & 31;
        const int32_t s0 = __shfl_sync(kFull, g, 7), s1 = __shfl_sync(kFull, g, 22);
        const bool shared = __popc(__ballot_sync(kFull, g >= 0 && g == s0)) > 3 || __popc(__ballot_sync(kFull, g >= 0 && g == s1)) > 3;
        const unsigned peers = shared ? __match_any_sync(kFull, g >= 0 ? g : -2 - lane) : 1u << lane;
        const int first = __ffs(peers) - 1;
        int32_t old = -1;
        if (g >= 0 && lane == first) old = atomicExch(head + g, v);
        old = __shfl_sync(kFull, old, first);
        const unsigned above = lane < 31 ? peers >> (lane + 1) : 0u;
        if (t < n) {
            __stcs(next + v, above ? v + __ffs(above) : old);
            if (BATCH) gparent[v] = g;
        }
    }
}

// Every link must ascend. The first to see one of a family that does not takes the family (its bit in
// `seen`) and puts it on its block's list; the block sorts those together (one thread each), so that
// the few walks do not hold up warps that are checking: 2^24 nodes of a random tree 0.19 -> 0.06 ms.
// Threads that check may read links being rewritten; whatever they see, they find the bit set.
constexpr int kCheckThreads = 256;
constexpr int kCheckIlp = 4;

__device__ void sort_family(int32_t p, int32_t n, int32_t *head, int32_t *next, uint32_t *heavy, int32_t *heavy_count) {
    int32_t kids[kLight];
    int k = 0;
    int32_t c = __ldcg(head + p);
    for (; c >= 0 && c < n && k < kLight; ++k) {  // insertion into ascending order
        int i = k;
        for (; i > 0 && kids[i - 1] > c; --i) kids[i] = kids[i - 1];
        kids[i] = c;
        c = __ldcg(next + c);
    }
    if (c >= 0) {  // too many for one thread
        atomicOr(heavy + (p >> 5), 1u << (p & 31));
        atomicAdd(heavy_count, 1);
        return;
    }
    head[p] = kids[0];
    for (int i = 0; i < k; ++i) next[kids[i]] = i + 1 < k ? kids[i + 1] : -1;
}

__global__ void __launch_bounds__(kCheckThreads)
    k_check_children(const int32_t *__restrict__ par, int32_t n, int32_t *head, int32_t *next,
                     uint32_t *__restrict__ seen, uint32_t *__restrict__ heavy, int32_t *__restrict__ heavy_count) {
    pdl_prologue();
    constexpr int kTile = kCheckThreads * kCheckIlp;
    __shared__ int32_t todo[2 * kTile];
    __shared__ int count;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const int64_t step = int64_t(gridDim.x) * kTile;
    for (int64_t base = int64_t(blockIdx.x) * kTile; base < n; base += step) {
        int32_t x[kCheckIlp];
#pragma unroll
        for (int j = 0; j < kCheckIlp; ++j) {
            const int64_t t = base + j * kCheckThreads + threadIdx.x;
            x[j] = t < n ? __ldcg(next + t) : -1;
        }
#pragma unroll
        for (int j = 0; j < kCheckIlp; ++j) {
            const int64_t t = base + j * kCheckThreads + threadIdx.x;
            if (x[j] < 0 || x[j] > t) continue;
            const int32_t p = par[t];
            const uint32_t bit = 1u << (p & 31);
            if (p >= 0 && p < n && !(atomicOr(seen + (p >> 5), bit) & bit)) todo[atomicAdd(&count, 1)] = p;
        }
        __syncthreads();
        const int found = count;
        if (found > kTile || base + step >= n) {
            for (int i = threadIdx.x; i < found; i += kCheckThreads) sort_family(todo[i], n, head, next, heavy, heavy_count);
            __syncthreads();
            if (threadIdx.x == 0) count = 0;
        }
        __syncthreads();
    }
}

// Up to kSortAll nodes nearly every family is pushed by threads that run together and has to be sorted, and
// what counts is the chain of dependent steps. Every node walks its family's list itself: the least larger
// label is its next sibling, and the least of all the first child. No marks, no second stage, and no
// insertions one after another. Results go to arrays of their own, so that nothing read changes (and L1
// serves the walks of siblings). Bound by the latency of the longest list: random tree of 2^16 nodes 8.7 us
// (k_check_children 18.3), of 2^18 11 (20), of 2^19 14 (22), families of 30 27 and 58 (62, 72); a path, which
// has nothing to sort, 8.6 and 10.4 (6.2, 6.0). Beyond, the work grows with the squares of the families: 2^20
// random 23 (23), families of 30 119 (61).
constexpr int32_t kSortAll = 1 << 19;

__global__ void __launch_bounds__(kCheckThreads)
    k_sort_children(const int32_t *__restrict__ par, int32_t n, const int32_t *__restrict__ head,
                    const int32_t *__restrict__ next, int32_t *__restrict__ head2, int32_t *__restrict__ next2,
                    uint32_t *__restrict__ heavy, int32_t *__restrict__ heavy_count) {
    pdl_prologue();
    const int64_t t = gtid();
    if (t >= n) return;
    if (head[t] < 0) head2[t] = -1;
    const int32_t p = par[t], first = p >= 0 && p < n ? __ldg(head + p) : -1;
    int32_t c = first, after = INT_MAX, least = INT_MAX;
    for (int k = 0; c >= 0 && c < n && k < kLight; ++k) {
        least = min(least, c);
        if (c > t) after = min(after, c);
        c = __ldg(next + c);
    }
    next2[t] = after < INT_MAX ? after : -1;
    if (c >= 0) {  // too many for one thread: k_sort_heavy writes all of the family's links
        if (first == t) {
            atomicOr(heavy + (p >> 5), 1u << (p & 31));
            atomicAdd(heavy_count, 1);
        }
    } else if (least == t) {
        head2[p] = int32_t(t);
    }
}

// ------------------------------------------------------------ long families out of order

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / kWarp;
constexpr int kRadix = 256;
static_assert(kThreads == kRadix, "the scatter handles one digit per thread");
// R = 32-element rounds per warp: a tile of 8 warps holds 256 * R elements (R = 8 or 16, the
// SORT_ROUNDS tuning knob; larger tiles give longer runs per digit in the scatter)

// lanes of the warp whose 8-bit digit equals this lane's, among the valid lanes (an invalid lane
// matches itself only): __match_any_sync, or eight ballots on the digit's bits
template <bool BALLOT>
__device__ __forceinline__ unsigned digit_peers(int d, bool valid, int lane) {
    if (!BALLOT) return __match_any_sync(kFull, valid ? d : kRadix + lane);
    unsigned peers = __ballot_sync(kFull, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1;
        const unsigned m = __ballot_sync(kFull, bit);
        peers &= bit ? m : ~m;
    }
    return valid ? peers : (1u << lane);
}

// A pass's histograms are 256 rows, one entry per block. Few blocks have many rows each, and short ones: there a
// warp takes a row, else a block. All passes, us, by blocks and by warps: stars of 5000 nodes (3 blocks) 119 and
// 37, 8193 (5) 70 and 35, 2^16 (32) 39 and 33, 2^18 (128) 46 and 48, 2^19 (257) 53 and 61.
constexpr int kShortRow = 64;

// all blocks of the cooperative grid; false (in every block that gets there) if the wait ran out
__device__ bool grid_barrier(uint32_t *bar, uint32_t target, int32_t *status) {
    constexpr int kPolls = 1 << 24;  // about ten seconds
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        int i = 0;
        while (*reinterpret_cast<volatile uint32_t *>(bar) < target && i < kPolls) {
            __nanosleep(100);
            ++i;
        }
        ok = i < kPolls;
        if (!ok) set_status(status, ETL_ETIMEOUT);
        __threadfence();
    }
    return __syncthreads_and(ok);
}

// Pairs (parent, child) of the heavy families in ascending child order, sorted by parent. Every block
// owns a contiguous part of a pass's input; ghist[digit * blocks + block] are the blocks' histograms.
template <int R, bool BALLOT>
__global__ void __launch_bounds__(kThreads)
    k_sort_heavy(const int32_t *__restrict__ par, int32_t n, const uint32_t *__restrict__ heavy,
                 const int32_t *__restrict__ heavy_count, int passes, int2 *buf0, int2 *buf1, int32_t *ghist,
                 int32_t *totals, uint32_t *bar, int32_t *__restrict__ head, int32_t *__restrict__ next, int32_t *__restrict__ status) {
    if (*heavy_count == 0) return;
    constexpr int kWarpTile = kWarp * R, kTile = kWarps * kWarpTile;
    __shared__ int32_t wcnt[kWarps][kRadix];
    __shared__ int32_t gbase[kRadix];   // next output place of each digit
    __shared__ int32_t dstart[kRadix];  // first tile position of each digit (digit order)
    __shared__ int32_t wtot[kWarps];
    __shared__ int2 stage[kTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = threadIdx.x;
    const int blocks = gridDim.x, blk = blockIdx.x;
    uint32_t arrivals = 0;
    int64_t count = n;  // of the pass's input: all nodes first, then the pairs kept
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        const int2 *in = p & 1 ? buf0 : buf1;
        int2 *out = p & 1 ? buf1 : buf0;
        const int64_t lo = count * blk / blocks, hi = count * (blk + 1) / blocks;
        auto load = [&](int64_t i) -> int2 {  // parent -1: not one of a heavy family
            if (i >= hi) return make_int2(-1, 0);
            if (p > 0) return __ldcg(in + i);
            const int32_t q = __ldg(par + i);
            const bool h = q >= 0 && q < n && ((__ldg(heavy + (q >> 5)) >> (q & 31)) & 1u);
            return make_int2(h ? q : -1, int32_t(i));
        };
        gbase[d] = 0;
        __syncthreads();
        for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) {
            const int32_t k = load(i).x;
            if (k >= 0) atomicAdd(&gbase[(k >> shift) & (kRadix - 1)], 1);
        }
        __syncthreads();
        ghist[int64_t(d) * blocks + blk] = gbase[d];
        arrivals += blocks;
        if (!grid_barrier(bar, arrivals, status)) return;
        // exclusive prefixes over the blocks, one digit's row at a time; its total goes to totals
        if (blocks <= kShortRow) {
            for (int row = blk * kWarps + warp; row < kRadix; row += blocks * kWarps) {
                int32_t carry = 0;
                for (int b0 = 0; b0 < blocks; b0 += kWarp) {
                    int32_t *at = ghist + int64_t(row) * blocks + b0 + lane;
                    const int32_t c = b0 + lane < blocks ? __ldcg(at) : 0;
                    int32_t inc = c;
#pragma unroll
                    for (int o = 1; o < kWarp; o <<= 1) {
                        const int32_t y = __shfl_up_sync(kFull, inc, o);
                        if (lane >= o) inc += y;
                    }
                    if (b0 + lane < blocks) *at = carry + inc - c;
                    carry += __shfl_sync(kFull, inc, kWarp - 1);
                }
                if (lane == 0) totals[row] = carry;
            }
        } else {
            for (int row = blk; row < kRadix; row += blocks) {
                int32_t carry = 0;
                for (int b0 = 0; b0 < blocks; b0 += kThreads) {
                    const int b = b0 + threadIdx.x;
                    int32_t *at = ghist + int64_t(row) * blocks + b;
                    const int32_t c = b < blocks ? __ldcg(at) : 0;
                    int32_t inc = c;
#pragma unroll
                    for (int o = 1; o < kWarp; o <<= 1) {
                        const int32_t y = __shfl_up_sync(kFull, inc, o);
                        if (lane >= o) inc += y;
                    }
                    if (lane == kWarp - 1) wtot[warp] = inc;
                    __syncthreads();
                    int32_t wofs = carry;
                    for (int w = 0; w < kWarps; ++w) {
                        if (w < warp) wofs += wtot[w];
                        carry += wtot[w];
                    }
                    if (b < blocks) *at = wofs + inc - c;
                    __syncthreads();
                }
                if (threadIdx.x == 0) totals[row] = carry;
            }
        }
        arrivals += blocks;
        if (!grid_barrier(bar, arrivals, status)) return;
        const int32_t all = __ldcg(totals + d), before = __ldcg(ghist + int64_t(d) * blocks + blk);
        int32_t inc = all;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == kWarp - 1) wtot[warp] = inc;
        __syncthreads();
        int32_t wofs = 0, total = 0;
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) wofs += wtot[w];
            total += wtot[w];
        }
        gbase[d] = wofs + inc - all + before;
        __syncthreads();
        for (int64_t base = lo; base < hi; base += kTile) {
            for (int w = 0; w < kWarps; ++w) wcnt[w][d] = 0;
            __syncthreads();
            int2 x[R];
            int32_t dig[R], lrank[R];
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = load(base + warp * kWarpTile + r * kWarp + lane);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool valid = x[r].x >= 0;
                const int dd = valid ? ((x[r].x >> shift) & (kRadix - 1)) : 0;
                const unsigned peers = digit_peers<BALLOT>(dd, valid, lane);
                int pre = 0;
                if (valid) pre = wcnt[warp][dd];
                __syncwarp();
                if (valid && lane == __ffs(peers) - 1) wcnt[warp][dd] = pre + __popc(peers);
                __syncwarp();
                dig[r] = valid ? dd : -1;
                lrank[r] = pre + __popc(peers & lanemask_lt());
            }
            __syncthreads();
            // counts of the warps -> offsets across warps; the digits' totals -> offsets across digits
            int32_t run = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const int32_t c = wcnt[w][d];
                wcnt[w][d] = run;
                run += c;
            }
            int32_t scan = run;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const int32_t y = __shfl_up_sync(kFull, scan, o);
                if (lane >= o) scan += y;
            }
            if (lane == kWarp - 1) wtot[warp] = scan;
            __syncthreads();
            int32_t ofs = 0, placed = 0;
            for (int w = 0; w < kWarps; ++w) {
                if (w < warp) ofs += wtot[w];
                placed += wtot[w];
            }
            dstart[d] = ofs + scan - run;
            __syncthreads();
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (dig[r] >= 0) stage[dstart[dig[r]] + wcnt[warp][dig[r]] + lrank[r]] = x[r];
            __syncthreads();
            for (int i = threadIdx.x; i < placed; i += kThreads) {
                const int2 y = stage[i];
                const int dd = (y.x >> shift) & (kRadix - 1);
                out[gbase[dd] + (i - dstart[dd])] = y;
            }
            __syncthreads();
            gbase[d] += run;
        }
        count = total;
        arrivals += blocks;
        if (!grid_barrier(bar, arrivals, status)) return;
    }
    const int2 *kv = passes & 1 ? buf0 : buf1;
    for (int64_t i = gtid(); i < count; i += gstride()) {
        const int2 x = __ldcg(kv + i);
        const int32_t before = i > 0 ? __ldcg(&kv[i - 1].x) : -1;
        const int2 y = i + 1 < count ? __ldcg(kv + i + 1) : make_int2(-1, -1);
        next[x.y] = y.x == x.x ? y.y : -1;
        if (before != x.x) head[x.x] = x.y;
    }
}

template <int R, bool BALLOT>
etl_status sort_heavy(const int32_t *par, int32_t n, const uint32_t *heavy, const int32_t *heavy_count, uint32_t *bar,
                      int32_t *head, int32_t *next, int32_t *status, Workspace &ws) {
    auto kernel = k_sort_heavy<R, BALLOT>;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0) != cudaSuccess || per_sm < 1)
        return ETL_ECUDA;
    // all that are resident at once on the stream's SMs, but no more than there are tiles
    const int64_t tiles = ceil_div(n, kWarps * kWarp * R), resident = int64_t(stream_sms(ws.stream())) * per_sm;
    const int blocks = int(tiles < resident ? tiles : resident);
    int2 *buf0 = ws.get<int2>(n), *buf1 = ws.get<int2>(n);
    int32_t *ghist = ws.get<int32_t>(int64_t(kRadix) * (blocks + 1)), *totals = ghist + int64_t(kRadix) * blocks;
    if (!ws.ok()) return ETL_ENOMEM;
    const int bits = ceil_log2(uint64_t(n));
    int passes = bits <= 8 ? 1 : (bits + 7) / 8;
    PhaseTimer pt("lca.heavy", ws.stream());
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks;
    cfg.blockDim = kThreads;
    cfg.stream = ws.stream();
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, par, n, heavy, heavy_count, passes, buf0, buf1, ghist, totals, bar, head, next, status);
    note_launch();
    return last_launch();
}

}  // namespace

SortParams &sort_params() {
    static SortParams p;
    return p;
}

etl_status link_children(const int32_t *parent, int32_t n, const int32_t *off, int32_t k, const int32_t *bad, int32_t *gparent,
                         int32_t *&head, int32_t *&next, int32_t *root_cnt, int32_t *root_of, int32_t *words, int32_t *status, Workspace &ws) {
    cudaStream_t s = ws.stream();
    const int64_t mask_words = ceil_div(n, 32);  // words: seen, heavy, heavy families, barrier
    uint32_t *seen = reinterpret_cast<uint32_t *>(words), *heavy = seen + mask_words, *bar = seen + 2 * mask_words + 1;
    int32_t *heavy_count = words + 2 * mask_words;
    const int32_t *par = off ? gparent : parent;
    {
        PhaseTimer pt("lca.link", s);
        const int64_t tiles = ceil_div(n, kLinkThreads * kLinkIlp);
        const int groups = off ? std::max(1, std::min(k / 8, kLinkGroups)) : 1;
        const int blocks = int(ceil_div(tiles, groups) * groups);
        launch(off ? k_link_children<true> : k_link_children<false>, blocks, kLinkThreads, 0, s, parent, n, groups, off, k,
               bad, gparent, head, next, root_cnt, root_of, status);
        note_launch();
    }
    {
        PhaseTimer pt("lca.check", s);
        if (n <= kSortAll) {
            int32_t *head2 = ws.get<int32_t>(n), *next2 = ws.get<int32_t>(n);
            if (!ws.ok()) return ETL_ENOMEM;
            launch(k_sort_children, int(ceil_div(n, kCheckThreads)), kCheckThreads, 0, s, par, n, head, next, head2, next2,
                   heavy, heavy_count);
            head = head2;
            next = next2;
        } else {
            const int64_t blocks = ceil_div(n, kCheckThreads * kCheckIlp), most = int64_t(num_sms()) * 8;
            launch(k_check_children, int(blocks < most ? blocks : most), kCheckThreads, 0, s, par, n, head, next, seen, heavy,
                   heavy_count);
        }
        note_launch();
    }
    etl_status st = last_launch();
    if (st || n <= kLight) return st;
    const SortParams &P = sort_params();
    if (P.rounds == 16)
        return P.ballot ? sort_heavy<16, true>(par, n, heavy, heavy_count, bar, head, next, status, ws)
                        : sort_heavy<16, false>(par, n, heavy, heavy_count, bar, head, next, status, ws);
    return P.ballot ? sort_heavy<8, true>(par, n, heavy, heavy_count, bar, head, next, status, ws)
                    : sort_heavy<8, false>(par, n, heavy, heavy_count, bar, head, next, status, ws);
}

}  // namespace etl
