// Internal declarations of the Euler-tour library (sm_103a). Not part of the ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "etl.h"

#define ETL_END (-1)

namespace etl {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// ----------------------------------------------------------------- host helpers

// Number of SMs of the current device (cached per device).
int num_sms();

// Number of SMs the work of a stream can use: fewer than the device has if the stream belongs to a green
// context. A cooperative grid must fit them: a larger one is refused at its launch, and replayed from a graph
// it would wait for ever.
int stream_sms(cudaStream_t s);

// Caller-owned device memory. While an ArenaScope is active on the calling
// thread, every device allocation the library makes (dev_alloc, and so
// Workspace::get and the tables of an LCA handle) is carved from the arena
// instead of the allocator: 256-byte aligned, never freed, never reused within
// the call. A measuring arena has no memory behind it: it hands out placeholder
// addresses and only counts bytes; it is used with a stream under capture, so
// the kernels that receive those addresses are recorded and never run, and the
// async memset / copy helpers below skip their work.
struct Arena {
    char *base = nullptr;  // caller's memory (null while measuring)
    size_t cap = 0;        // bytes available from base
    size_t used = 0;       // bytes handed out so far (alignment included)
    bool measure = false;
};
Arena *current_arena();
class ArenaScope {
  public:
    explicit ArenaScope(Arena *a);
    ~ArenaScope();
    ArenaScope(const ArenaScope &) = delete;
    ArenaScope &operator=(const ArenaScope &) = delete;

  private:
    Arena *prev_;
};
inline bool measuring() {
    const Arena *a = current_arena();
    return a && a->measure;
}

// Stream-ordered device allocation from the library's own per-device memory
// pool, which keeps freed memory reserved (release threshold = max) so that
// repeated calls do not pay for re-mapping, and never reuses a block freed on
// another stream by making this stream wait for that one; while the stream is
// being captured into a graph the default pool is used (graph memory nodes).
// Freed with cudaFreeAsync. Inside an ArenaScope the memory comes from the
// arena instead (and must not be freed). Returns cudaSuccess or the
// allocator's error (cudaErrorMemoryAllocation when the arena is too small).
cudaError_t dev_alloc(void **p, size_t bytes, cudaStream_t s);

// cudaMemsetAsync / device-to-device cudaMemcpyAsync, skipped while measuring
cudaError_t memset_async(void *p, int value, size_t bytes, cudaStream_t s);
cudaError_t copy_d2d_async(void *dst, const void *src, size_t bytes, cudaStream_t s);

// Stream-ordered scratch: released with cudaFreeAsync on the same stream when the Workspace goes out of
// scope. Small buffers are cut from chunks, so that a call on a small input asks the allocator for memory
// once or twice and not for each of its dozen buffers (1 us of host time for each pair of calls); buffers
// in a caller's arena are cut from that one by one.
class Workspace {
  public:
    explicit Workspace(cudaStream_t s) : s_(s), arena_(current_arena() != nullptr) {}
    ~Workspace() { release(); }
    Workspace(const Workspace &) = delete;
    Workspace &operator=(const Workspace &) = delete;
    template <class T>
    T *get(size_t count) {
        size_t bytes = count * sizeof(T);
        if (bytes == 0) bytes = 16;
        if (arena_ || bytes > kSmall) return static_cast<T *>(take(bytes));
        bytes = (bytes + 255) & ~size_t(255);
        if (bytes > left_) {
            at_ = static_cast<char *>(take(kChunk));
            left_ = at_ ? kChunk : 0;
            if (!at_) return nullptr;
        }
        char *p = at_;
        at_ += bytes;
        left_ -= bytes;
        return reinterpret_cast<T *>(p);
    }
    bool ok() const { return ok_; }
    void release() {
        if (!arena_)
            for (void *p : bufs_) cudaFreeAsync(p, s_);
        bufs_.clear();
        left_ = 0;
    }
    cudaStream_t stream() const { return s_; }

  private:
    static constexpr size_t kChunk = size_t(4) << 20, kSmall = size_t(1) << 20;
    void *take(size_t bytes) {
        void *p = nullptr;
        if (dev_alloc(&p, bytes, s_) != cudaSuccess) {
            ok_ = false;
            return nullptr;
        }
        bufs_.push_back(p);
        return p;
    }
    cudaStream_t s_;
    std::vector<void *> bufs_;
    char *at_ = nullptr;  // rest of the current chunk
    size_t left_ = 0;
    bool ok_ = true;
    bool arena_;  // buffers come from a caller-owned arena: nothing to free
};

// Brackets a launch group with CUDA events when phase timing is enabled
// (etl_profile_enable); a no-op otherwise and while the stream is captured.
class PhaseTimer {
  public:
    PhaseTimer(const char *name, cudaStream_t s);
    ~PhaseTimer();
    PhaseTimer(const PhaseTimer &) = delete;
    PhaseTimer &operator=(const PhaseTimer &) = delete;

  private:
    const char *name_;
    cudaStream_t s_;
    void *a_ = nullptr, *b_ = nullptr;
};

// Host-side count of kernel launches issued by the library (for reporting).
void note_launch();

inline etl_status last_launch() {
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ETL_OK : ETL_ECUDA;
}

// Programmatic dependent launch (ETL_TUNE_PDL). Every kernel of the library starts with
// pdl_prologue(): it waits until the grid launched before it on the stream has finished and its
// writes are visible (a no-op when the kernel was not launched as a dependent), then allows the
// next grid on the stream to be scheduled. launch() issues a kernel with the attribute when the knob
// is on, so the next kernel's launch overlaps the end of the current one instead of following it.
bool &pdl_enabled();

__device__ __forceinline__ void pdl_prologue() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline void launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Args &&>(args)...);
}

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

inline int ceil_log2(uint64_t x) {  // smallest b with 2^b >= x (x >= 1)
    int b = 0;
    while ((uint64_t(1) << b) < x) ++b;
    return b;
}

// ----------------------------------------------------------------- device helpers

__device__ __forceinline__ void set_status(int32_t *st, int32_t code) {
    if (st) atomicCAS(st, 0, code);
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// largest i in [lo, hi] with off[i] <= x (off ascending, off[lo] <= x)
__device__ __forceinline__ int32_t last_at_or_before(const int32_t *__restrict__ off, int32_t lo, int32_t hi, int64_t x) {
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo + 1) >> 1);
        if (__ldg(off + mid) <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// ----------------------------------------------------------------- primitives

// Exclusive scan of in[0..n) into out[0..n], out[n] = total.
etl_status scan_exclusive_i32(const int32_t *in, int32_t *out, int64_t n, Workspace &ws);

// Children of every node in ascending label order: head[v] = first child or -1, next[c] = next sibling
// or -1 (-1 for roots too). parent: ids in [0, n), -1 at roots; anything else is dropped and sets the
// status. For a batch of k instances, off (k + 1 offsets; *bad: unusable, drop all nodes) says which one a
// node belongs to, ids are local to it, and gparent receives the global ones (-1 at roots, -2: dropped).
// The caller has set head to -1 and cleared root_cnt, root_of (roots per instance and the last one seen) and
// words (link_words(n) of them, scratch). head and next may come back as other arrays of the workspace.
inline int64_t link_words(int64_t n) { return 2 * ((n + 31) / 32) + 2; }
etl_status link_children(const int32_t *parent, int32_t n, const int32_t *off, int32_t k, const int32_t *bad, int32_t *gparent,
                         int32_t *&head, int32_t *&next, int32_t *root_cnt, int32_t *root_of, int32_t *words, int32_t *status, Workspace &ws);

// ----------------------------------------------------------------- list ranking

// Records of ranked list elements: the sublist's id, the element's offset in it (lr) and, in 8-byte
// records, the number of even-indexed elements before it in the sublist (lo; bit 15 of that field: a
// contracted leaf). In the in-place form (rank.cu) the same word is the element's slot: its successor
// before the ranking, its record afterwards. A slot can also be marked as not on the list: a walk that
// comes across it by claiming it at random leaves it alone.
struct Slot4 {  // successor < 2^30 or -1; kOff; record: top bit, sublist id << lb, lr (never -1)
    using T = uint32_t;
    static constexpr uint32_t kOff = 0x7ffffffeu;
    __device__ static __forceinline__ T exch(T *p, T v) { return atomicExch(p, v); }
    __device__ static __forceinline__ bool off(T v) { return v == kOff; }
    __device__ static __forceinline__ bool raw(T v) { return (!(v >> 31) && v != kOff) || v == 0xffffffffu; }
    __device__ static __forceinline__ T make(int32_t succ) { return uint32_t(succ); }
    __device__ static __forceinline__ T off_list() { return kOff; }
    __device__ static __forceinline__ int32_t next(T v) { return int32_t(v); }
    __device__ static __forceinline__ T rec(int32_t sid, uint32_t lr, uint32_t, int lb) {
        return 0x80000000u | (uint32_t(sid) << lb) | lr;
    }
    __device__ static __forceinline__ int32_t sid(T v, int lb) { return int32_t((v & 0x7fffffffu) >> lb); }
    __device__ static __forceinline__ uint32_t lr(T v, int lb) { return v & ((1u << lb) - 1u); }
};
struct Slot8 {  // low word: successor / sublist id; high word: kRaw / kOff / lr | lo << 16
    using T = unsigned long long;
    static constexpr uint32_t kRaw = 0xffffffffu, kOff = 0xfffffffeu;
    __device__ static __forceinline__ T pack(uint32_t lo, uint32_t hi) { return (T(hi) << 32) | lo; }
    __device__ static __forceinline__ T exch(T *p, T v) { return atomicExch(p, v); }
    __device__ static __forceinline__ bool off(T v) { return uint32_t(v >> 32) == kOff; }
    __device__ static __forceinline__ bool raw(T v) { return uint32_t(v >> 32) == kRaw; }
    __device__ static __forceinline__ T make(int32_t succ) { return pack(uint32_t(succ), kRaw); }
    __device__ static __forceinline__ T off_list() { return pack(uint32_t(ETL_END), kOff); }
    __device__ static __forceinline__ int32_t next(T v) { return int32_t(uint32_t(v)); }
    __device__ static __forceinline__ T rec(int32_t sid, uint32_t lr, uint32_t lo, int) {
        return pack(uint32_t(sid), lr | (lo << 16));
    }
    __device__ static __forceinline__ int32_t sid(T v, int) { return int32_t(uint32_t(v)); }
    __device__ static __forceinline__ uint32_t lr(T v, int) { return uint32_t(v >> 32) & 0xffffu; }
    __device__ static __forceinline__ uint32_t lo(T v) { return uint32_t(v >> 48) & 0x7fffu; }
    __device__ static __forceinline__ bool leaf(T v) { return (v >> 63) && !raw(v) && !off(v); }
};
// 4-byte slots of a tour (dual) with fewer than 2^29 elements: successor, bit 30: contracted leaf; -1;
// kOff; record: top bit, sublist id (22 bits), lr (lr + 1) / 2 + lo (9 bits: lr < kLcap, lo <= lr). Short
// sublists, but half the memory of 8-byte slots.
struct Slot4d {
    using T = uint32_t;
    static constexpr uint32_t kOff = 0x7ffffffeu;
    static constexpr int kLcap = 31, kSidBits = 22;
    __device__ static __forceinline__ T exch(T *p, T v) { return atomicExch(p, v); }
    __device__ static __forceinline__ bool off(T v) { return v == kOff; }
    __device__ static __forceinline__ bool raw(T v) { return (!(v >> 31) && v != kOff) || v == 0xffffffffu; }
    __device__ static __forceinline__ T make(int32_t succ) {  // leaf: top bit set
        return succ < ETL_END ? (uint32_t(succ) & 0x3fffffffu) | 0x40000000u : uint32_t(succ);
    }
    __device__ static __forceinline__ T off_list() { return kOff; }
    __device__ static __forceinline__ int32_t next(T v) {
        return v == 0xffffffffu ? ETL_END : int32_t((v & 0x40000000u) ? (v & 0x3fffffffu) | 0x80000000u : v);
    }
    __device__ static __forceinline__ T rec(int32_t sid, uint32_t lr, uint32_t lo, int) {
        return 0x80000000u | (uint32_t(sid) << 9) | (((lr * (lr + 1)) >> 1) + lo);
    }
    __device__ static __forceinline__ int32_t sid(T v, int) { return int32_t((v & 0x7fffffffu) >> 9); }
    __device__ static __forceinline__ uint32_t lr(T v, int) {
        const uint32_t k = v & 511u;
        return uint32_t((sqrtf(float(8u * k + 1u)) - 1.0f) * 0.5f);  // exact: the root of a perfect square is
    }
    __device__ static __forceinline__ uint32_t lo(T v, uint32_t lr) { return (v & 511u) - ((lr * (lr + 1)) >> 1); }
};
inline bool wide_slots(int64_t len) { return len > (int64_t(1) << 30); }

// Result of ranking one list: element e's record names its sublist; first[sid], or in dual mode
// first2[sid].x / .y, are the number of elements / of even-indexed elements before that sublist's first
// element. So rank(e) = first + lr and evens_before(e) = first2.y + lo.
struct RankResult {
    const void *recs;  // Slot8 records if wide; else Slot4 or, in dual mode, Slot4d ones
    bool wide;
    int lb;
    const int32_t *first;
    const int2 *first2;
    int64_t rcap;  // sublists
};

// rank of element e of a list ranked without dual; -1 if its record shows that it is not on the list
__device__ __forceinline__ int32_t rank_at(const RankResult &r, int64_t e) {
    int32_t sid, lr;
    if (r.wide) {
        const Slot8::T v = static_cast<const Slot8::T *>(r.recs)[e];
        if (Slot8::raw(v) || Slot8::off(v)) return -1;
        sid = Slot8::sid(v, 0);
        lr = int32_t(Slot8::lr(v, 0));
    } else {
        const Slot4::T v = static_cast<const Slot4::T *>(r.recs)[e];
        if (Slot4::raw(v) || Slot4::off(v)) return -1;
        sid = Slot4::sid(v, r.lb);
        lr = int32_t(Slot4::lr(v, r.lb));
    }
    return (sid >= 0 && sid < r.rcap) ? __ldg(r.first + sid) + lr : -1;
}

struct RankParams {
    int k0_log2 = 5;     // level-0 splitter density: one in 2^k0_log2 elements
    int k_log2 = 3;      // density at the upper levels (1 in 8: 1-4% faster than 1 in 16 on trees of 2^15 .. 2^22)
    int block = 128;     // threads per block of the walk kernels
    int blocks_per_sm = 10;  // 1280 walkers per SM on lists ranked in place
};
RankParams &rank_params();

struct SortParams {
    int rounds = 8;       // 32-element rounds per warp in the radix passes over long families: tiles of 256 * rounds
    bool ballot = true;   // rank equal digits in a warp by ballots instead of __match_any_sync
};
SortParams &sort_params();

struct CcParams {
    int first_slice_quarters = 2;  // edges hooked before the first compression, in units of n/4
    bool doubling = false;         // later slices double in size, each after a compression
    bool giant = true;             // after a compression, the most frequent root ranks above all
};
CcParams &cc_params();

struct RmqParams {
    int levels_per_pass = 3;  // 1..3 levels built by one streaming pass
    int block = 256;          // threads per block of the level kernel
    bool blocked = true;      // two-level (blocked) tables instead of full sparse tables
};
RmqParams &rmq_params();

// What list_rank takes: int32 successors (the records get an array of their own), or slots that the
// records replace (8-byte slots: Slot8; 4-byte ones: Slot4, in dual mode Slot4d).
enum class RankForm { kSeparate, kSlots8, kSlots4 };
RankForm rank_form(int64_t len, bool dual);
// Ranks a list of len elements in that form, from *d_head, or from `head` if d_head is null. An element
// that is on no list holds off_list() in a slot, Slot4::kOff as a successor; a contracted leaf's second
// element off_list() in a slot, -1 as a successor. dual: also counts even-indexed elements (the opening
// brackets of a tour). expect_len: the total weight the list must have (-1: not checked). zero: a device
// word that is zero when this runs and is not used afterwards (or null: the call clears one itself).
etl_status list_rank(void *list, int64_t len, const int32_t *d_head, int32_t head, bool dual, int64_t expect_len,
                     int32_t *zero, int32_t *status, Workspace &ws, RankResult *out);

// ----------------------------------------------------------------- sparse tables

// Full sparse table over x[0..n): level l holds min (or max) of x[i .. i+2^l)
// (entries past the end are folded with the identity). levels =
// floor(log2(max_len)) + 1 where max_len is the longest range ever queried.
// Level 0 must already be in table[0..n); rows are sparse_ld(n) apart and the
// build pads each row's tail with the identity.
int sparse_levels(int64_t max_len);
// row length (entries) of a table over n entries: n rounded up to a multiple of 4
int64_t sparse_ld(int64_t n);
template <bool IS_MAX>
etl_status sparse_table_build(int32_t *table, int64_t n, int levels, cudaStream_t s);

template <bool IS_MAX>
__device__ __forceinline__ int32_t sparse_query(const int32_t *__restrict__ table, int64_t ld, int32_t lo,
                                                int32_t hi) {  // inclusive range, lo <= hi; ld = row length
    int len = hi - lo + 1;
    int l = 31 - __clz(len);
    const int32_t *t = table + int64_t(l) * ld;
    int32_t a = __ldg(t + lo), b = __ldg(t + hi - (1 << l) + 1);
    return IS_MAX ? max(a, b) : min(a, b);
}

// ----------------------------------------------------------------- blocked range-min / max tables
//
// Two levels over x[0..n): x is cut into blocks of 32 entries; pm[i] / sm[i]
// hold op over x from the start of i's block to i / from i to the end of its
// block, and `top` is a full sparse table over the nblk block results. A range
// [lo, hi] inside one block is answered from x directly (at most 32 entries of
// one 128-byte line); otherwise it is op(sm[lo], pm[hi]) plus, when whole
// blocks lie between, one query of `top`. The build reads x once and writes
// 2n + O(n / 32 * log n) entries; `top` (n / 32 entries per level) stays in L2.
// Layout of one allocation of element type T: x, pm, sm (nblk * 32 entries
// each, x padded with the identity by the build) then tlevels rows of `top`,
// nblk entries apart.

struct OpMin {
    using T = int32_t;
    __device__ static __forceinline__ T id() { return INT32_MAX; }
    __device__ static __forceinline__ T f(T a, T b) { return min(a, b); }
};
struct OpMinKey {  // 64-bit keys: a value in the high half, a payload it carries in the low half
    using T = long long;
    __device__ static __forceinline__ T id() { return INT64_MAX; }
    __device__ static __forceinline__ T f(T a, T b) { return min(a, b); }
};
struct OpMinMax {  // x = min of the first component, y = max of the second
    using T = int2;
    __device__ static __forceinline__ T id() { return make_int2(INT32_MAX, INT32_MIN); }
    __device__ static __forceinline__ T f(T a, T b) { return make_int2(min(a.x, b.x), max(a.y, b.y)); }
};

constexpr int kRmqBlockLog2 = 5;
constexpr int kRmqBlock = 1 << kRmqBlockLog2;

struct BlockedLayout {
    int64_t nblk;  // blocks of 32 entries
    int tlevels;   // levels of the top table
    int64_t elems() const { return 3 * nblk * kRmqBlock + nblk * tlevels; }
};
// a table over n entries answering ranges of up to max_len entries
BlockedLayout blocked_layout(int64_t n, int64_t max_len);
// x (first n entries of base) must be filled; builds pad, pm, sm and top
template <class Op>
etl_status blocked_build(typename Op::T *base, int64_t n, const BlockedLayout &L, cudaStream_t s);
// the top table from its first row. (A handle's table has pm and sm interleaved as (pm[i], sm[i]) pairs in
// the 2N entries after x, built in lca.cu: blocked_query, which reads them as separate arrays, is not for it.)
template <class Op>
etl_status blocked_top(typename Op::T *top, const BlockedLayout &L, cudaStream_t s);

template <class Op>
struct BlockedView {
    const typename Op::T *x, *pm, *sm, *top;
    int64_t nblk;
    int tlevels;
};
template <class Op>
inline BlockedView<Op> blocked_view(const typename Op::T *base, const BlockedLayout &L) {
    const int64_t N = L.nblk * kRmqBlock;
    return BlockedView<Op>{base, base + N, base + 2 * N, base + 3 * N, L.nblk, L.tlevels};
}
// longest range a layout answers (a range of len entries spans at most (len - 1) / 32 whole blocks)
inline int64_t blocked_max_len(const BlockedLayout &L) { return (int64_t(kRmqBlock) << L.tlevels) - 1; }

template <class Op>
__device__ __forceinline__ typename Op::T blocked_query(const BlockedView<Op> &t, int32_t lo,
                                                        int32_t hi) {  // inclusive, lo <= hi
    using T = typename Op::T;
    const int32_t bl = lo >> kRmqBlockLog2, bh = hi >> kRmqBlockLog2;
    if (bl == bh) {
        T m = __ldg(t.x + lo);
        for (int32_t j = lo + 1; j <= hi; ++j) m = Op::f(m, __ldg(t.x + j));
        return m;
    }
    T m = Op::f(__ldg(t.sm + lo), __ldg(t.pm + hi));
    if (bh - bl > 1) {
        const int32_t a = bl + 1, b = bh - 1;
        const int l = 31 - __clz(b - a + 1);
        const T *row = t.top + int64_t(l) * t.nblk;
        m = Op::f(m, Op::f(__ldg(row + a), __ldg(row + b - (1 << l) + 1)));
    }
    return m;
}

}  // namespace etl

// ----------------------------------------------------------------- the LCA handle
struct etl_lca_s {
    int32_t n = 0;       // nodes (all instances of a batch together)
    int32_t k = 1;       // trees in the handle
    int32_t *node_off = nullptr;  // batch only: k+1 instance offsets (device)
    int levels = 0;
    cudaStream_t stream = nullptr;
    int32_t *pre = nullptr, *depth = nullptr, *size = nullptr, *order = nullptr;
    int64_t ld = 0;             // row length of the sparse table
    int32_t *table = nullptr;   // levels * ld (full sparse table) or the blocked table's allocation
    bool blocked = false;       // table is a blocked two-level table (layout `bl`)
    void *nrec = nullptr;       // blocked table: per node (pre, pm[pre], sm[pre], size), int4[n]
    etl::BlockedLayout bl{};
    int32_t *status = nullptr;  // device status word
    bool has_table = false;     // RMQ sparse table built (lca_query available)
    void *inrec = nullptr;      // Inlabel: per node (inlabel, ascendant, depth, parent), int4[n]
    void *inpath = nullptr;     // Inlabel: per inlabel value (parent of the path head, its depth), int2[n+1]
    void *tour_table = nullptr;  // Euler-tour RMQ: blocked table of (depth << 32 | node) keys over 2n positions
    int32_t *tpos = nullptr;     // Euler-tour RMQ: tour position of each node's opening bracket
    etl::BlockedLayout tbl{};
    void *block = nullptr;       // the allocation that pre .. order, table, nrec, status and node_off are cut from
    bool arena = false;          // device arrays live in a caller-owned workspace: lca_free frees none of them
};

namespace etl {
// Single trees of up to kTinyNodes nodes with the blocked table (or none): all of the preprocessing in one
// launch (tiny.cu; 8192 nodes 36 us with their queries, apart 52, beyond the shared memory runs out).
constexpr int kTinyNodes = 8192;
etl_status build_tiny_tree(const int32_t *parent, etl_lca_s *h, cudaStream_t s);
}  // namespace etl
