// Ranking of a list in the shared memory of one block: the top of the list ranker's recursion (rank.cu)
// and the tours of small trees (tiny.cu).
#pragma once

#include "etl_internal.cuh"

namespace etl {

constexpr int kTopThreads = 1024;
constexpr int kTopCap = 15360;         // entries (12 bytes each)
constexpr int kTopSub = kTopThreads;   // sublists
constexpr int32_t kEndT = 0x7fffffff;  // "no successor" in a reduced list's entry
constexpr int32_t kVisited = int32_t(0x80000000u);

constexpr uint32_t kHashMul = 0x9E3779B1u;  // odd, so multiplication is a bijection mod 2^b

constexpr uint32_t inverse_mod_2_32(uint32_t a) {  // Newton iteration for a^-1 mod 2^32 (a odd)
    uint32_t x = a;
    for (int i = 0; i < 5; ++i) x *= 2u - a * x;
    return x;
}

// Splitters of a list: element e is one iff its hash is below S0; the hash is the sublist's id.
struct Hash {
    uint32_t mask, S0;  // elements [0, mask]
    __device__ __forceinline__ bool split(uint32_t e) const { return ((e * kHashMul) & mask) < S0; }
    __device__ __forceinline__ int32_t sid(uint32_t e) const { return int32_t((e * kHashMul) & mask); }
    __device__ __forceinline__ uint32_t elem(uint32_t s) const {
        constexpr uint32_t kInv = inverse_mod_2_32(kHashMul);
        return (s * kInv) & mask;
    }
};

struct TopShared {
    int32_t QF[kTopSub], V1[kTopSub], V2[kTopSub];
    int found;
};

// Called by a block of kTopThreads after nx (successor, kEndT or anything >= len: none), a1 and a2 (the
// weights; a2 with DUAL only) of all len entries are in shared memory and a barrier has passed. At most
// kTopSub - 1 splitters and the head cut the list into sublists, one per thread, which are walked and then
// ranked by pointer jumping: Q = predecessor, F = first sublist of the segment from there, V1 / V2 = sums
// over the segment (Q, e]. A round replaces Q and F by the predecessor's and adds its segment; after
// ceil(log2 kTopSub) rounds every Q is none and V is the inclusive prefix from the list's first sublist F.
// After it (ends with a barrier) an entry that was walked has its sublist's id and the top bit in nx and
// its offsets in a1, a2; the prefixes before the sublists are in V1, V2. Bound by shared memory: a step
// reads and writes two or three random words, and a round three random ones per sublist; with 2048
// sublists, two to a thread, the walks took the same time and the rounds twice theirs (15360 entries,
// dual: 31 us before, 26 now).
template <bool DUAL>
__device__ __forceinline__ void rank_in_shared(int len, int32_t head, int64_t expect_total, TopShared &sh, int32_t *nx,
                                               int32_t *a1, int32_t *a2, int32_t *status) {
    Hash H;
    const int b = len <= 1 ? 0 : 32 - __clz(len - 1);
    H.mask = (1u << b) - 1u;
    H.S0 = min((H.mask + 1u) >> 1, uint32_t(kTopSub - 1));
    const bool head_split = H.split(uint32_t(head));
    const int32_t head_sub = head_split ? H.sid(uint32_t(head)) : int32_t(H.S0);
    const int w = threadIdx.x;
    int32_t e = w < int(H.S0) ? int32_t(H.elem(uint32_t(w))) : w == int(H.S0) && !head_split ? head : len;
    int32_t s1 = 0, s2 = 0, link = kEndT;
    while (e >= 0 && e < len) {
        const int32_t z = nx[e], y1 = a1[e], y2 = DUAL ? a2[e] : 0;
        if (z < 0) {  // visited before: no list
            set_status(status, ETL_EBADTREE);
            break;
        }
        nx[e] = kVisited | w;
        a1[e] = s1;
        if (DUAL) a2[e] = s2;
        s1 += y1;
        s2 += y2;
        e = z;
        if (z < len && H.split(uint32_t(z))) {
            link = H.sid(uint32_t(z));
            break;
        }
    }
    sh.QF[w] = w << 16;  // (F, Q + 1)
    sh.V1[w] = s1;
    sh.V2[w] = s2;
    if (w == 0) sh.found = 0;
    __syncthreads();
    if (link != kEndT) sh.QF[link] = (link << 16) | (w + 1);  // a link is a sublist id below kTopSub
    __syncthreads();
    int32_t qf = sh.QF[w], v1 = s1, v2 = s2;
    for (int rounds = 0;; ++rounds) {
        const int32_t q = (qf & 0xffff) - 1;
        if (q >= 0) {
            qf = sh.QF[q];
            v1 += sh.V1[q];
            if (DUAL) v2 += sh.V2[q];
        }
        if (!__syncthreads_or(q >= 0)) break;
        if (rounds > 40) {  // a cycle: cannot happen on a valid list
            if (w == 0) set_status(status, ETL_EBADTREE);
            break;
        }
        sh.QF[w] = qf;
        sh.V1[w] = v1;
        if (DUAL) sh.V2[w] = v2;
        __syncthreads();
    }
    if (expect_total >= 0 && link == kEndT && (qf >> 16) == head_sub && int64_t(v1) == expect_total) sh.found = 1;
    sh.V1[w] = v1 - s1;  // exclusive
    sh.V2[w] = v2 - s2;
    __syncthreads();
    if (w == 0 && expect_total >= 0 && !sh.found) set_status(status, ETL_EBADTREE);
}

}  // namespace etl
