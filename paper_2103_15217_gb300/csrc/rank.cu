// List ranking on the GPU (Sec. 2.2): the successor array of the Euler tour is
// ranked once, and every later prefix sum over the tour is taken from these
// ranks. The paper uses the Wei-JaJa sparse-ruling-set method; this is a
// GB300-oriented ruling-set ranker:
//
//  * Level 0 cuts the list into sublists, walks them and leaves a record
//    (sublist id, local offset) per element. It has two forms:
//    - k_walk0, for tours of up to 2^22 brackets and other lists whose
//      successors and records fit in L2: sublists start at splitters picked
//      by a multiplicative hash of the element index, e is one iff
//      (e * M mod 2^b) < S0; the hashed value is the sublist's id. A step is one dependent load, 0.25 us, and the walks are
//      bound by the longest sublist, about len / S0 * ln S0 steps.
//    - k_walk0_in_place, for longer ones, which are bound by memory (tours by
//      the rate of L2 first, of DRAM from some 2^25 brackets on): element and
//      record share one slot, and a step is ONE atomic exchange, which
//      stores the record and returns the successor. Reading the successor in
//      one array and writing the record in another touches two sectors per
//      element over three times the memory: 2^25 random elements take 1.65 ms
//      that way (4 B read + 8 B write) and 0.49 ms as 4-byte exchanges (0.95
//      ms as 8-byte ones), measured with independent accesses. An exchange
//      takes 0.47 us, so the short lists keep the loads. (A load followed by
//      a store to the same sector costs 1 us and more.)
//  * The in-place form decides where sublists start as it runs. Every lane
//    claims an element by exchanging it for the record (its sublist, offset 0)
//    and walks on from there; a walk ends at the tail or where its exchange
//    returns another walk's record, which it puts back and links to. A lane
//    whose walk has ended claims its next candidate; if that was visited
//    already, the record goes back and the claim is dropped. So long sublists
//    are cut by the lanes that have run out of work: with 13 claims per lane
//    the last walk ends after 2 to 2.5 len / lanes steps, and 2.5 to 3 sublists
//    per lane have been opened. Candidates are the multiples of the golden
//    ratio times len (any prefix of them is evenly spread, and no two of
//    len / 3 fall on one element).
//  * A walk whose offset no longer fits the record opens a new sublist and
//    goes on in it ("dynamic" sublist).
//  * The reduced list of sublists (weights = sublist length, and number of
//    even-indexed elements) is cut and walked again until at most kTopCap
//    entries are left, which one CTA ranks in shared memory: walks, then
//    pointer jumping over at most kTopSub sublists. The prefixes are pushed
//    back down level by level.
//
// The "dual" mode also counts even-indexed elements: in the bracket layout
// of a rooted tree (2v = entering v, 2v+1 = leaving v) that count is the
// preorder number, so preorder comes straight out of the ranking without a
// scatter + scan over the tour. In dual mode a successor with the top bit
// set (and not -1) marks a contracted leaf: element 2v of a leaf v stands for
// both of its brackets (weight 2), the low 31 bits are the successor of 2v+1,
// and 2v+1 itself is off the list.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "rank_top.cuh"

namespace etl {
namespace {

constexpr int32_t kLcap = 4096;  // longest sublist of 8-byte records (< 2^15)
// candidate w >= 1 of a list of len elements: floor(frac(w * golden ratio) * len). The distance of any
// two of the first W multiples is above 0.38 / W, so W <= len / 3 candidates are distinct elements.
__device__ __forceinline__ int64_t candidate(uint32_t w, int64_t len) {
    return int64_t(__umul64hi(uint64_t(w) * 0x9E3779B97F4A7C15ull, uint64_t(len)));
}

// A warp's supply of sublist ids: kFirst of its own, then kTake at a time from a counter. Only a
// successful claim uses one up, so that the reduced list has few empty entries; once the ids have passed
// `limit` the warp claims nothing any more (claims shorten the walks; the result does not need them).
// (Ids 8 at a time, all from the counter: the walk of 2^25 elements 10% slower, each refill holds up the
// warp for one contended atomic.)
struct SidPool {
    static constexpr int kFirst = 64, kTake = 32;
    int32_t base, count;  // the same in every lane
    bool closed = false;
    __device__ __forceinline__ explicit SidPool(uint32_t warp) : base(int32_t(warp) * kFirst), count(kFirst) {}
    // ids from the counter start at `start`
    __device__ __forceinline__ void refill(int32_t *ctr, int32_t start, int32_t limit, bool need, int32_t &sid) {
        const unsigned m = __ballot_sync(kFull, need);
        if (!m) return;
        const int cnt = __popc(m), i = __popc(m & lanemask_lt());
        int32_t nb = 0;
        const bool more = cnt > count;
        if (more) {
            if ((threadIdx.x & 31) == 0) nb = start + atomicAdd(ctr, kTake);
            nb = __shfl_sync(kFull, nb, 0);
            closed = nb + kTake > limit;
        }
        if (need) sid = i < count ? base + i : nb + (i - count);
        if (more) {
            base = nb + (cnt - count);
            count += kTake - cnt;
        } else {
            base += cnt;
            count -= cnt;
        }
    }
    // ids taken and not used become empty sublists
    __device__ __forceinline__ void give_back(int32_t sid, int4 *T, int32_t cap) const {
        if (sid >= 0 && sid < cap) T[sid] = make_int4(0, 0, kEndT, 0);
        for (int i = threadIdx.x & 31; i < count; i += kWarp)
            if (base + i < cap) T[base + i] = make_int4(0, 0, kEndT, 0);
    }
};

// *d_len entries (plus those of *d_add), at most cap
__device__ __forceinline__ int64_t level_len(int64_t base, const int32_t *d_add, int64_t cap) {
    return min(base + (d_add ? int64_t(*d_add) : 0), cap);
}

// ------------------------------------------------------------ level-0 walk over a list in L2

// Sublist ids: a splitter's hash, S0 for the head's own sublist, S0 + 1 + d for dynamic ones. A lane
// takes the ids w, w + lanes, ... A record is written once the successor is known, so that it can say
// whether the element is a contracted leaf.
template <class S, bool DUAL>
__global__ void k_walk0(const uint32_t *__restrict__ succ, int64_t len, const int32_t *__restrict__ d_head,
                        int32_t head_value, Hash H, typename S::T *__restrict__ recs, int lb, uint32_t lcap,
                        int4 *__restrict__ T, int32_t *__restrict__ dyn, int32_t cap, int32_t *__restrict__ next_head,
                        int32_t *__restrict__ status) {
    pdl_prologue();
    const int32_t head = d_head ? *d_head : head_value;
    const bool head_split = H.split(uint32_t(head));
    const uint32_t nwork = H.S0 + 1, lanes = gridDim.x * blockDim.x;
    uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w == 0) *next_head = head_split ? H.sid(uint32_t(head)) : int32_t(H.S0);
    int32_t cur = -1, sid = 0;
    uint32_t lr = 0, lo = 0;
    int64_t steps = 0;
    while (true) {
        if (cur < 0) {
            if (w >= nwork) break;
            const int64_t e = w < H.S0 ? int64_t(H.elem(w)) : head_split ? len : int64_t(head);
            sid = int32_t(w);
            w += lanes;
            if (e < 0 || e >= len) {  // no element behind this id
                T[sid] = make_int4(0, 0, kEndT, 0);
                continue;
            }
            cur = int32_t(e);
            lr = lo = 0;
            steps = 0;
        }
        const uint32_t v = __ldg(succ + cur);
        int32_t nxt = int32_t(v);
        bool leaf = false;
        if (DUAL && nxt < ETL_END) {  // contracted leaf: its closing bracket follows at once
            nxt &= 0x7fffffff;
            leaf = true;
        }
        recs[cur] = S::rec(sid, lr, leaf ? lo | 0x8000u : lo, lb);
        const uint32_t l0 = lr;
        lr += leaf ? 2 : 1;
        if (DUAL) lo += (cur & 1) == 0 ? 1u : 0u;
        int32_t link = kEndT;
        if (nxt == ETL_END) {
            cur = -1;
        } else if (nxt < 0 || nxt >= len || ++steps > len) {
            // a slot that is off the list may be a splitter; reaching one is an error
            if (v != Slot4::kOff || l0) set_status(status, ETL_EBADTREE);
            if (v == Slot4::kOff && !l0) lr = 0;
            cur = -1;
        } else if (H.split(uint32_t(nxt))) {
            link = H.sid(uint32_t(nxt));
            cur = -1;
        } else {
            cur = nxt;
            if (lr >= lcap) {
                const int32_t ns = int32_t(H.S0) + 1 + atomicAdd(dyn, 1);
                if (ns >= cap) {
                    set_status(status, ETL_ETIMEOUT);
                    cur = -1;
                } else {
                    T[sid] = make_int4(int32_t(lr), int32_t(lo), ns, 0);
                    sid = ns;
                    lr = lo = 0;
                }
            }
        }
        if (cur < 0) T[sid] = make_int4(int32_t(lr), int32_t(lo), link, 0);
    }
}

// ------------------------------------------------------------ level-0 walk in place

struct Walk0 {
    int64_t len;
    const int32_t *d_head;  // the list's head, or null: `head`
    int32_t head;
    uint32_t nclaims;  // the head and nclaims - 1 candidates
    int32_t start;     // sublist ids below it belong to the warps, the counter hands out those above
    int32_t limit;     // ids after which no more claims are made
    int32_t cap;       // sublists there is room for
    int32_t lb;        // 4-byte records: bits of the local offset
    int32_t lcap;      // a sublist of lcap elements is continued in a new one
};

// One lane = one walk at a time. The claims of a lane are fixed (its index, + lanes, + 2 lanes, ...),
// so that no counter is shared by them.
template <class S, bool DUAL>
__global__ void k_walk0_in_place(typename S::T *__restrict__ slots, Walk0 W, int4 *__restrict__ T, int32_t *__restrict__ ctr,
                        int32_t *__restrict__ next_head, int32_t *__restrict__ status) {
    pdl_prologue();
    const uint32_t lanes = gridDim.x * blockDim.x;
    uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t head = W.d_head ? *W.d_head : W.head;
    SidPool pool(w >> 5);
    int32_t cur = -1, sid = -1;
    uint32_t lr = 0, lo = 0;
    bool active = false, claim = false, is_head = false;
    while (true) {
        const bool want = !active && w < W.nclaims, full = active && lr >= uint32_t(W.lcap);
        int32_t ns = sid;
        pool.refill(ctr, W.start, W.limit, (want && sid < 0) || full, ns);
        if (full) {  // the walk goes on in a new sublist
            if (ns < W.cap) {
                T[sid] = make_int4(int32_t(lr), int32_t(lo), ns, 0);
                lr = lo = 0;
            } else {
                set_status(status, ETL_ETIMEOUT);
                T[sid] = make_int4(int32_t(lr), int32_t(lo), kEndT, 0);
                active = false;
                ns = -1;
            }
        }
        sid = ns;
        if (want) {
            is_head = w == 0;
            const int64_t e = is_head ? int64_t(head) : candidate(w, W.len);
            w += lanes;
            if (sid < W.cap && e >= 0 && e < W.len) {  // both always hold; keep memory safe
                cur = int32_t(e);
                lr = lo = 0;
                active = claim = true;
            }
        }
        if (pool.closed) w = W.nclaims;
        if (!__any_sync(kFull, active)) {
            if (!__any_sync(kFull, w < W.nclaims)) break;
            continue;
        }
        if (!active) continue;
        const typename S::T v = S::exch(slots + cur, S::rec(sid, lr, lo, W.lb));
        int32_t link = kEndT;
        bool done = false;
        if (!S::raw(v)) {  // visited already, or off the list: put it back
            S::exch(slots + cur, v);
            if (claim) {
                if (is_head) *next_head = S::off(v) ? 0 : S::sid(v, W.lb);
                if (S::off(v) && is_head) set_status(status, ETL_EBADTREE);
                active = false;
            } else {  // link to the sublist that starts here
                if (S::off(v) || S::lr(v, W.lb) != 0)
                    set_status(status, ETL_EBADTREE);  // not the first of a sublist: a second predecessor
                else
                    link = S::sid(v, W.lb);
                done = true;
            }
        } else {
            if (claim && is_head) *next_head = sid;
            claim = false;
            int32_t nxt = S::next(v);
            lr += 1;
            if (DUAL) {
                lo += (cur & 1) == 0 ? 1u : 0u;
                if (nxt < ETL_END) {  // contracted leaf: its closing bracket follows at once
                    nxt &= 0x7fffffff;
                    lr += 1;
                }
            }
            if (nxt == ETL_END) {
                done = true;
            } else if (nxt < 0 || nxt >= W.len) {
                set_status(status, ETL_EBADTREE);
                done = true;
            } else {
                cur = nxt;
            }
        }
        if (done) {
            T[sid] = make_int4(int32_t(lr), int32_t(lo), link, 0);
            active = false;
            sid = -1;
        }
    }
    pool.give_back(sid, T, W.cap);
}

// ------------------------------------------------------------ upper-level walk (explicit weights)

// Entry of a reduced list: x, y = the sublist's weights, z = the id of the next sublist (kEndT: none).
// The hash covers the entries there are (the device knows how many); one in 2^k_log2 is a splitter, and
// never more than `most`. One 16-byte load per step, 0.25 us; an entry's place (sublist, offsets) goes to
// loc. (Replacing the entry by it would put a load and a store on one sector.) A walk is as long as its
// sublist: nothing cuts it short, and nothing has to, as the sums are 32 bits wide.
__global__ void k_walk(const int4 *__restrict__ T, int64_t base, const int32_t *__restrict__ d_add, int64_t cap,
                       const int32_t *__restrict__ d_head, int k_log2, uint32_t most, int4 *__restrict__ loc,
                       int4 *__restrict__ up, int32_t *__restrict__ up_len, int32_t *__restrict__ next_head,
                       int32_t *__restrict__ status) {
    pdl_prologue();
    const int64_t len = level_len(base, d_add, cap);
    const int32_t head = *d_head;
    Hash H;
    const int b = len <= 1 ? 0 : 64 - __clzll(len - 1);
    H.mask = (1u << b) - 1u;
    H.S0 = min(((H.mask >> k_log2) + 1u), most);
    const bool head_split = H.split(uint32_t(head));
    const uint32_t nwork = H.S0 + 1, lanes = gridDim.x * blockDim.x;
    uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w == 0) {
        *next_head = head_split ? H.sid(uint32_t(head)) : int32_t(H.S0);
        *up_len = int32_t(nwork);
    }
    int32_t cur = -1, sid = 0, a1 = 0, a2 = 0;
    int64_t steps = 0;
    while (true) {
        if (cur < 0) {
            if (w >= nwork) break;
            const int64_t e = w < H.S0 ? int64_t(H.elem(w)) : head_split ? len : int64_t(head);
            sid = int32_t(w);
            w += lanes;
            if (e < 0 || e >= len) {
                up[sid] = make_int4(0, 0, kEndT, 0);
                continue;
            }
            cur = int32_t(e);
            a1 = a2 = 0;
            steps = 0;
        }
        const int4 t = __ldg(T + cur);
        loc[cur] = make_int4(a1, a2, sid, 0);
        a1 += t.x;
        a2 += t.y;
        int32_t link = kEndT;
        if (t.z == kEndT) {
            cur = -1;
        } else if (t.z < 0 || t.z >= len || ++steps > len) {
            set_status(status, ETL_EBADTREE);
            cur = -1;
        } else if (H.split(uint32_t(t.z))) {
            link = H.sid(uint32_t(t.z));
            cur = -1;
        } else {
            cur = t.z;
        }
        if (cur < 0) up[sid] = make_int4(a1, a2, link, 0);
    }
}

// ------------------------------------------------------------ top level: one CTA, shared memory

// The sums before an entry. They have an array of their own, 8 or 4 bytes per entry, not the first half of
// the 16-byte entries: the top writes half the sectors, and what is gathered from it later stays small.
template <bool DUAL>
using Prefix = std::conditional_t<DUAL, int2, int32_t>;
template <bool DUAL>
__device__ __forceinline__ Prefix<DUAL> prefix(int32_t x, int32_t y) {
    if constexpr (DUAL)
        return make_int2(x, y);
    else
        return x;
}

// FROM_LIST: the list itself instead of a reduced list; each element on it becomes its own sublist in
// the result. One SM issues all of it, so the steps are kept to a few instructions (claims as in the
// in-place walk, tried here, took twice the time; pointer jumping over all entries three times).
constexpr int kTopBatch = 5;  // entries per thread whose loads are in flight together

template <class S, bool DUAL, bool FROM_LIST>
__global__ void __launch_bounds__(kTopThreads)
    k_top(const uint32_t *__restrict__ succ, typename S::T *__restrict__ recs, int lb, const int4 *__restrict__ T,
          Prefix<DUAL> *__restrict__ out, int64_t base, const int32_t *__restrict__ d_add, int64_t cap, const int32_t *__restrict__ d_head,
          int32_t head_value, int64_t expect_total, int32_t *__restrict__ status) {
    pdl_prologue();
    extern __shared__ int32_t sm[];
    __shared__ TopShared sh;
    const int len = int(level_len(base, d_add, cap));
    int32_t *nx = sm, *a1 = nx + len, *a2 = a1 + len;
    const int32_t head = d_head ? *d_head : head_value;
    for (int i = threadIdx.x; i < len; i += kTopBatch * kTopThreads) {
        int4 t[kTopBatch];
        uint32_t v[kTopBatch];
#pragma unroll
        for (int j = 0; j < kTopBatch; ++j) {
            const int e = i + j * kTopThreads;
            if (e < len) {
                if (FROM_LIST)
                    v[j] = succ[e];
                else
                    t[j] = T[e];
            }
        }
#pragma unroll
        for (int j = 0; j < kTopBatch; ++j) {
            const int e = i + j * kTopThreads;
            if (e >= len) continue;
            if (FROM_LIST) {
                int32_t nxt = int32_t(v[j]), w1 = 1;
                if (DUAL && nxt < ETL_END) {
                    nxt &= 0x7fffffff;
                    w1 = 2;
                }
                // anything that is no element ends the list (the total is checked)
                nx[e] = (nxt < 0 || nxt >= len) ? kEndT : nxt;
                a1[e] = w1;
                if (DUAL) a2[e] = (e & 1) == 0 ? 1 : 0;
                if (nxt != ETL_END && nxt >= len && v[j] != Slot4::kOff) set_status(status, ETL_EBADTREE);
                if (!DUAL && nxt < ETL_END) set_status(status, ETL_EBADTREE);
                if (!DUAL && expect_total >= 0 && v[j] == Slot4::kOff) set_status(status, ETL_EBADTREE);
            } else {
                nx[e] = t[j].z;
                a1[e] = t[j].x;
                if (DUAL) a2[e] = t[j].y;
            }
        }
    }
    __syncthreads();
    rank_in_shared<DUAL>(len, head, expect_total, sh, nx, a1, a2, status);
    for (int e = threadIdx.x; e < len; e += kTopThreads) {
        const int32_t z = nx[e], w = z & (kTopSub - 1);
        const bool on = z < 0;  // on a walk
        out[e] = prefix<DUAL>(on ? sh.V1[w] + a1[e] : 0, DUAL && on ? sh.V2[w] + a2[e] : 0);
        if (FROM_LIST && on) {
            const bool leaf = DUAL && int32_t(succ[e]) < ETL_END;
            recs[e] = S::rec(e, 0, leaf ? 0x8000u : 0u, lb);
        }
    }
}

size_t top_smem(int64_t len, bool dual) { return size_t((dual ? 3 : 2) * len) * sizeof(int32_t); }

// an entry's prefix over the whole list: its sublist's and that in the sublist
template <bool DUAL>
__global__ void k_expand(const int4 *__restrict__ loc, int64_t base, const int32_t *__restrict__ d_add, int64_t cap,
                         const Prefix<DUAL> *__restrict__ up, int64_t up_cap, Prefix<DUAL> *__restrict__ out) {
    pdl_prologue();
    const int64_t len = level_len(base, d_add, cap);
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < len; e += int64_t(gridDim.x) * blockDim.x) {
        const int4 l = __ldcs(loc + e);
        if (l.z < 0 || l.z >= up_cap) continue;  // entries on no walk get whatever is there
        if constexpr (DUAL) {
            const int2 u = __ldg(up + l.z);
            out[e] = make_int2(u.x + l.x, u.y + l.y);
        } else {
            out[e] = __ldg(up + l.z) + l.x;
        }
    }
}

// succ -> slots of the in-place walk
template <class S>
__global__ void k_list_slots(const int32_t *succ, int64_t len, typename S::T *slots) {
    pdl_prologue();
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < len; e += int64_t(gridDim.x) * blockDim.x)
        slots[e] = S::make(__ldcs(succ + e));
}

// rank and 4-byte records may be the same array
__global__ void k_final_rank(RankResult rr, int64_t len, int32_t *rank) {
    pdl_prologue();
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < len; e += int64_t(gridDim.x) * blockDim.x)
        rank[e] = rank_at(rr, e);
}

}  // namespace

RankParams &rank_params() {
    static RankParams p;
    return p;
}

// Shorter lists keep successors and records in separate arrays, longer ones are ranked in place, in 4-byte
// slots where the records fit them. Tours of random trees, whole ranking: 2^21 brackets 139 us apart, 139
// in place, 2^22 183 and 182, 2^23 250 and 226. Other lists: 2^22 elements 173 and 182, 2^23 251 and 233,
// but a caller's list has to be copied into the slots first, so the line lies where successors and records
// (8 bytes per element) exceed 96 of the 129 MB of L2.
RankForm rank_form(int64_t len, bool dual) {
    if (dual ? len <= (int64_t(1) << 22) : len * 8 <= (int64_t(96) << 20)) return RankForm::kSeparate;
    if (dual) return len <= (int64_t(1) << 26) ? RankForm::kSlots4 : RankForm::kSlots8;
    return wide_slots(len) ? RankForm::kSlots8 : RankForm::kSlots4;
}

namespace {

int grid_of(int64_t lanes, int64_t per_sm, const RankParams &P) {
    const int64_t most = int64_t(num_sms()) * (per_sm > 0 ? per_sm : 1);
    return int(std::max<int64_t>(1, std::min(most, ceil_div(lanes, P.block))));
}

// splitters of a level of len entries, one in 2^k of the hashed range; if that is at most twice the
// top's capacity, as many as the top takes (one level less, or shorter walks), but one in two at most
uint32_t splitters(int64_t len, int k) {
    const uint32_t range = uint32_t(uint64_t(1) << ceil_log2(uint64_t(len)));
    const uint32_t s = std::max(1u, range >> k);
    return s < 2u * kTopCap ? std::max(std::min(s, uint32_t(kTopCap - 1)), std::min(range >> 1, uint32_t(kTopCap - 1))) : s;
}

// A: where scratch comes from (get<T>(count); a null pointer when there is none). list: len 4-byte
// successors, recs: room for len records (or null: taken from alloc); in place: list = slots S::T. zero: a
// device word that is zero (or null)
template <class S, bool DUAL, class A>
etl_status rank_impl(void *list, void *recs, int64_t len, const int32_t *d_head, int32_t head, int64_t expect_len,
                     int32_t *zero, int32_t *status, const RankParams &P, A &alloc, cudaStream_t s, RankResult *out) {
    using R = typename S::T;
    const bool in_place = rank_form(len, DUAL) != RankForm::kSeparate;
    constexpr bool kNarrow = std::is_same<S, Slot4d>::value;
    // 4-byte slots of a tour and 8-byte ones of another list are only ever ranked in place
    constexpr bool kApart = DUAL ? !kNarrow : std::is_same<S, Slot4>::value;
    out->wide = sizeof(R) == 8;
    out->lb = out->wide ? 16 : 12;
    if (in_place) recs = list;
    if (!recs) recs = alloc.template get<R>(len);
    if (!recs) return ETL_ENOMEM;
    out->recs = recs;
    const uint32_t *succ = static_cast<const uint32_t *>(list);
    cudaFuncSetAttribute(k_top<S, DUAL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(top_smem(kTopCap, DUAL)));
    etl_status st = ETL_OK;
    auto set_result = [&](Prefix<DUAL> *first, int64_t cap) {
        if constexpr (DUAL)
            out->first2 = first;
        else
            out->first = first;
        out->rcap = cap;
    };
    if constexpr (kApart) {
        if (len <= kTopCap) {
            cudaFuncSetAttribute(k_top<S, DUAL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(top_smem(kTopCap, DUAL)));
            Prefix<DUAL> *first = alloc.template get<Prefix<DUAL>>(len);
            if (!first) return ETL_ENOMEM;
            set_result(first, len);
            PhaseTimer pt("rank.top", s);
            launch(k_top<S, DUAL, true>, 1, kTopThreads, top_smem(len, DUAL), s, succ, static_cast<R *>(recs), out->lb, nullptr,
                   first, len, nullptr, len, d_head, head, expect_len, status);
            note_launch();
            return last_launch();
        }
    }

    struct Level {
        int4 *T, *loc;
        Prefix<DUAL> *first;
        int64_t base, cap;  // entries: base + *d_add, at most cap
        const int32_t *d_add, *d_head;
    };
    Level lv[32];
    int nl = 0;
    int32_t *words = alloc.template get<int32_t>(64);  // per level: [2 i] entry count, [2 i + 1] head
    if (!words) return ETL_ENOMEM;
    if (!zero) {
        zero = words;
        memset_async(zero, 0, sizeof(int32_t), s);
    }
    if (in_place) {
        Walk0 w{};
        w.len = len;
        w.d_head = d_head;
        w.head = head;
        const int64_t per_lane = int64_t(2) << P.k0_log2;
        // two thirds of the walkers where the slots fit L2: 2^24 random brackets 304 us, 320 with all of them
        const bool fits = len * int64_t(sizeof(R)) <= (int64_t(96) << 20);
        const int grid = grid_of(len / per_lane, fits ? std::max(1, P.blocks_per_sm * 2 / 3) : P.blocks_per_sm, P);
        const int64_t lanes = int64_t(grid) * P.block;
        w.nclaims = uint32_t(std::min(16 * lanes, len / 3) + 1);
        w.start = int32_t(lanes / kWarp * SidPool::kFirst);
        // a warp may pass the limit once, by up to 32 ids, and has up to 31 left over in the end
        if (kNarrow) {
            w.lcap = Slot4d::kLcap;
            const int64_t most = (int64_t(1) << Slot4d::kSidBits) - 2 * lanes - (len / w.lcap + 2);
            w.limit = int32_t(std::min(8 * lanes, most));
            w.cap = int32_t(w.limit + 2 * lanes + len / w.lcap + 2);
        } else {
            // sublist id and local offset share 31 bits of a 4-byte record: the longest offset for which
            // they fit (8 bits for 2^30 elements)
            w.limit = int32_t(8 * lanes);
            for (w.lb = out->wide ? 16 : 12;; --w.lb) {
                w.lcap = out->wide ? kLcap : (1 << w.lb) - 1;
                w.cap = int32_t(w.limit + 2 * lanes + len / w.lcap + 2);
                if (out->wide || int64_t(w.cap) <= (int64_t(1) << (31 - w.lb)) || w.lb <= 4) break;
            }
        }
        out->lb = w.lb;
        int4 *T = alloc.template get<int4>(w.cap);
        if (!T) return ETL_ENOMEM;
        lv[nl++] = Level{T, nullptr, nullptr, w.start, w.cap, zero, words + 1};
        PhaseTimer pt0("rank.walk0_in_place", s);
        launch(k_walk0_in_place<S, DUAL>, grid, P.block, 0, s, static_cast<R *>(recs), w, T, zero, words + 1, status);
        note_launch();
        st = last_launch();
    } else if constexpr (kApart) {
        const int k = std::min(P.k0_log2, len > (int64_t(1) << 20) ? 4 : 3);
        Hash H;
        H.mask = uint32_t((uint64_t(1) << ceil_log2(uint64_t(len))) - 1);
        uint32_t lcap;
        int32_t dyn_cap, cap;
        for (;; --out->lb) {  // as above
            lcap = out->wide ? uint32_t(kLcap) : (1u << out->lb) - 1u;
            dyn_cap = int32_t(len / lcap + 2);
            H.S0 = splitters(len, k);
            // ids of dynamic sublists come out of the same power of two, so that the next level's hash
            // does not cover twice the entries
            H.S0 -= std::min(H.S0 / 2, uint32_t(dyn_cap) + 1);
            cap = int32_t(H.S0) + 1 + dyn_cap;
            if (out->wide || int64_t(cap) <= (int64_t(1) << (31 - out->lb)) || out->lb <= 4) break;
        }
        int4 *T = alloc.template get<int4>(cap);
        if (!T) return ETL_ENOMEM;
        lv[nl++] = Level{T, nullptr, nullptr, int64_t(H.S0) + 1, cap, zero, words + 1};
        PhaseTimer pt0(DUAL ? "rank.walk0" : "rank.walk0_list", s);
        launch(k_walk0<S, DUAL>, grid_of(int64_t(H.S0) + 1, 2048 / P.block, P), P.block, 0, s, succ, len, d_head, head,
               H, static_cast<R *>(recs), out->lb, lcap, T, zero, cap, words + 1, status);
        note_launch();
        st = last_launch();
    } else {
        st = ETL_EINVAL;  // never: see kApart
    }
    if (st) return st;

    // ---- upper levels until one CTA can finish the reduced list
    while (lv[nl - 1].cap > kTopCap) {
        Level &L = lv[nl - 1];
        uint32_t most = splitters(L.cap, P.k_log2);
        if (most >= uint32_t(kTopCap)) --most;  // with the head's sublist, a power of two again
        L.loc = alloc.template get<int4>(L.cap);
        int4 *up = alloc.template get<int4>(int64_t(most) + 1);
        if (!L.loc || !up || nl >= 32) return ETL_ENOMEM;
        {
            PhaseTimer ptw("rank.walk", s);
            launch(k_walk, grid_of(int64_t(most) + 1, 2048 / P.block, P), P.block, 0, s, L.T, L.base, L.d_add, L.cap,
                   L.d_head, most < uint32_t(kTopCap) ? 0 : P.k_log2, most, L.loc, up, words + 2 * nl,
                   words + 2 * nl + 1, status);
            note_launch();
            st = last_launch();
        }
        if (st) return st;
        lv[nl] = Level{up, nullptr, nullptr, 0, int64_t(most) + 1, words + 2 * nl, words + 2 * nl + 1};
        ++nl;
    }

    for (int i = 0; i < nl; ++i)
        if (!(lv[i].first = alloc.template get<Prefix<DUAL>>(lv[i].cap))) return ETL_ENOMEM;
    // ---- top
    {
        const Level &L = lv[nl - 1];
        PhaseTimer ptp("rank.top", s);
        launch(k_top<S, DUAL, false>, 1, kTopThreads, top_smem(L.cap, DUAL), s, nullptr, nullptr, 0, L.T, L.first, L.base,
               L.d_add, L.cap, L.d_head, 0, expect_len, status);
        note_launch();
        st = last_launch();
        if (st) return st;
    }
    // ---- push prefixes back down
    for (int i = nl - 2; i >= 0; --i) {
        const Level &L = lv[i];
        int blocks = int(ceil_div(L.cap, 256));
        if (blocks > num_sms() * 32) blocks = num_sms() * 32;  // four waves of full occupancy
        PhaseTimer pte("rank.expand", s);
        launch(k_expand<DUAL>, blocks, 256, 0, s, L.loc, L.base, L.d_add, L.cap, lv[i + 1].first, lv[i + 1].cap, L.first);
        note_launch();
        st = last_launch();
        if (st) return st;
    }
    set_result(lv[0].first, lv[0].cap);
    return ETL_OK;
}

// The records take the place of the ranks, unless the caller's two arrays overlap: then records apart from the
// successors would overwrite them, and slots made from them in parallel would overwrite those of other threads
// (but not where rank is succ itself, when a thread writes only over what it has read).
template <class A>
etl_status rank_plain_list(const int32_t *succ, int64_t len, int32_t head, int32_t *rank, int32_t *status,
                           const RankParams &P, A &alloc, cudaStream_t s) {
    const bool wide = wide_slots(len), in_place = rank_form(len, false) != RankForm::kSeparate;
    const bool apart = succ < rank + len && rank < succ + len && !(in_place && succ == rank);
    void *recs = wide ? static_cast<void *>(alloc.template get<Slot8::T>(len))
                      : apart ? static_cast<void *>(alloc.template get<Slot4::T>(len)) : rank;
    if (!recs) return ETL_ENOMEM;
    int blocks = int(ceil_div(len, 256));
    if (blocks > num_sms() * 16) blocks = num_sms() * 16;
    void *list = const_cast<int32_t *>(succ);
    if (in_place) {
        PhaseTimer pt("rank.slots", s);
        if (wide)
            launch(k_list_slots<Slot8>, blocks, 256, 0, s, succ, len, static_cast<Slot8::T *>(recs));
        else
            launch(k_list_slots<Slot4>, blocks, 256, 0, s, succ, len, static_cast<Slot4::T *>(recs));
        note_launch();
        list = recs;
    }
    etl_status rc = last_launch();
    RankResult rr{};
    if (!rc)
        rc = wide ? rank_impl<Slot8, false>(list, recs, len, nullptr, head, len, nullptr, status, P, alloc, s, &rr)
                  : rank_impl<Slot4, false>(list, recs, len, nullptr, head, len, nullptr, status, P, alloc, s, &rr);
    if (rc) return rc;
    PhaseTimer pt("rank.final", s);
    launch(k_final_rank, blocks, 256, 0, s, rr, len, rank);
    note_launch();
    return last_launch();
}

}  // namespace

etl_status list_rank(void *list, int64_t len, const int32_t *d_head, int32_t head, bool dual, int64_t expect_len,
                     int32_t *zero, int32_t *status, Workspace &ws, RankResult *out) {
    cudaStream_t s = ws.stream();
    const RankParams &P = rank_params();
    if (dual && rank_form(len, true) == RankForm::kSlots4)
        return rank_impl<Slot4d, true>(list, nullptr, len, d_head, head, expect_len, zero, status, P, ws, s, out);
    if (dual) return rank_impl<Slot8, true>(list, nullptr, len, d_head, head, expect_len, zero, status, P, ws, s, out);
    if (wide_slots(len))
        return rank_impl<Slot8, false>(list, nullptr, len, d_head, head, expect_len, zero, status, P, ws, s, out);
    return rank_impl<Slot4, false>(list, nullptr, len, d_head, head, expect_len, zero, status, P, ws, s, out);
}

}  // namespace etl

extern "C" etl_status etl_list_rank(const int32_t *succ, int64_t len, int32_t head, int32_t *rank, int32_t *status,
                                    void *stream) {
    using namespace etl;
    if (!succ || !rank || len < 1 || len > int64_t(INT32_MAX) - 1 || head < 0 || head >= len) return ETL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Workspace ws(s);
    int32_t *st = status ? status : ws.get<int32_t>(1);
    if (!ws.ok()) return ETL_ENOMEM;
    return rank_plain_list(succ, len, head, rank, st, rank_params(), ws, s);
}

// ------------------------------------------------------------------ list ranking without allocation
//
// etl_list_rank_static: the same ranking as etl_list_rank, but every byte of
// scratch it needs comes from one fixed array of device memory that the
// library reserves when it is loaded, so the call itself never allocates.
// It exists for callers that cannot allocate device memory at the point of
// the call: code that runs under an external memory manager that owns the
// whole device (so a cudaMalloc would fail or fragment its arena), code that
// must not block on the allocator's implicit synchronisation, and code with a
// fixed, pre-planned memory budget. Such callers still pass their own input
// and output arrays.
//
// Limits and rules (also in etl.h):
//  * len <= kStaticMaxLen (2^18 elements); larger lists are rejected with
//    ETL_EINVAL before anything is enqueued.
//  * The scratch array (kStaticBytes, 3 MiB) is a file-scope __device__
//    variable: every GPU on which the library is loaded holds it until the
//    process exits.
//  * All calls share it and it keeps the previous call's contents; the
//    counters that must start at zero are cleared by each call. Two calls
//    whose work overlaps on the GPU (different streams, or different host
//    threads) race on the same scratch and give wrong ranks: serialise them.
//  * The host cannot use the array's name as a device address, so the first
//    call on each device looks the address up with cudaGetSymbolAddress (with
//    that device current) and caches it with the id of the CUDA context it
//    belongs to; that first call should therefore come before any stream
//    capture on that device. When the context changes (cudaDeviceReset, or
//    the primary context destroyed and made again), the next call sees the
//    new context id and repeats the look-up instead of using a stale address.
namespace etl {
namespace {

constexpr int64_t kStaticMaxLen = int64_t(1) << 18;
constexpr size_t kStaticBytes = size_t(3) << 20;

static __device__ __align__(256) unsigned char g_rank_scratch[kStaticBytes];

struct StaticArena {
    char *base;
    size_t used, cap;
    template <class T>
    T *get(int64_t count) {
        size_t off = (used + 255) & ~size_t(255);
        size_t bytes = size_t(count > 0 ? count : 1) * sizeof(T);
        if (off + bytes > cap) return nullptr;
        used = off + bytes;
        return reinterpret_cast<T *>(base + off);
    }
};

std::mutex g_static_mu;
void *g_static_addr[64] = {nullptr};
unsigned long long g_static_ctx[64] = {0};

// The driver's cuCtxGetCurrent / cuCtxGetId, reached through the runtime (no link against libcuda).
using CtxGetCurrentFn = int (*)(void **);
using CtxGetIdFn = int (*)(void *, unsigned long long *);
CtxGetCurrentFn g_ctx_get_current = nullptr;
CtxGetIdFn g_ctx_get_id = nullptr;
std::once_flag g_ctx_fns_once;

// id of the calling thread's current CUDA context (unique over the process's lifetime); false when
// there is no current context or the driver entry points are unavailable
bool current_context_id(unsigned long long *id) {
    std::call_once(g_ctx_fns_once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_ctx_get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_ctx_get_id = reinterpret_cast<CtxGetIdFn>(f);
    });
    if (!g_ctx_get_current || !g_ctx_get_id) return false;
    void *ctx = nullptr;
    if (g_ctx_get_current(&ctx) != 0 || !ctx) return false;
    return g_ctx_get_id(ctx, id) == 0;
}

// with the device current: the device address of the scratch array, looked up once per device and
// context (and again after the context changed)
etl_status static_scratch(void **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ETL_ECUDA;
    std::lock_guard<std::mutex> g(g_static_mu);
    // without the driver's context ids (entry points not found) the address is cached per device only
    unsigned long long id = 0;
    const bool have_id = current_context_id(&id);
    if (!g_static_addr[dev] || (have_id && g_static_ctx[dev] != id)) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_rank_scratch) != cudaSuccess || !p) return ETL_ECUDA;
        // the look-up made the device's primary context current if it was not yet
        g_static_ctx[dev] = current_context_id(&id) ? id : 0;
        g_static_addr[dev] = p;
    }
    *out = g_static_addr[dev];
    return ETL_OK;
}

}  // namespace
}  // namespace etl

extern "C" etl_status etl_list_rank_static(const int32_t *succ, int64_t len, int32_t head, int32_t *rank,
                                           int32_t *status, void *stream) {
    using namespace etl;
    if (!succ || !rank || len < 1 || head < 0 || head >= len) return ETL_EINVAL;
    if (len > kStaticMaxLen) return ETL_EINVAL;  // beyond the fixed scratch: documented limit
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void *scratch = nullptr;
    etl_status rc = static_scratch(&scratch);
    if (rc) return rc;
    StaticArena A{static_cast<char *>(scratch), 0, kStaticBytes};
    int32_t *st = status;
    if (!st) {
        st = A.get<int32_t>(1);
        if (cudaMemsetAsync(st, 0, sizeof(int32_t), s) != cudaSuccess) return ETL_ECUDA;
    }
    // fixed parameters, so that the layout is fixed (1.6 MB at the largest length; the slots are in the
    // caller's rank array)
    return rank_plain_list(succ, len, head, rank, st, RankParams{}, A, s);
}
