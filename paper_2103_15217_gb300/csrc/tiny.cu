// Preprocessing of a small tree in one launch: one block does every step of lca.cu in shared memory
// (children in label order, the tour's list, its ranking, preorder / depth / size, the blocked
// range-minimum table and the query records) and writes the handle's arrays. The steps take a few
// microseconds each whatever the size, and apart they are 13 launches: a tree of 1000 nodes took 44 us on
// the device and 60 us of host time for its launches and allocations, in one block 12 and 11.
#include <climits>

#include "rank_top.cuh"

namespace etl {
namespace {

// If there are families of more than kFamily children: labels from the highest down, 32 at a time by one warp (550
// cycles a step): lanes with the same parent form one run, which
// goes in front of the parent's list, so every list ascends.
constexpr int kFamily = 64;

__device__ void link_descending(const int32_t *par, int n, int32_t *head, int32_t *next2) {
    const int lane = threadIdx.x & 31;
    constexpr int kAhead = 4;  // loads of the next steps' parents, in flight during a step
    int32_t p[kAhead];
    const int top = (n - 1) & ~31;
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
        const int v = top - 32 * j + lane;
        p[j] = v >= 0 && v < n ? par[v] : -1;
    }
    for (int base = top; base >= 0; base -= 32 * kAhead) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int v = base - 32 * j + lane;
            const bool on = v >= 0 && v < n;
            const int32_t g = on ? p[j] : -1;
            const int ahead = v - 32 * kAhead;
            p[j] = ahead >= 0 ? par[ahead] : -1;
            const unsigned peers = __match_any_sync(kFull, g >= 0 ? g : -1 - lane);
            const unsigned above = lane < 31 ? peers >> (lane + 1) : 0u;
            const int32_t old = g >= 0 ? head[g] : -1;
            __syncwarp();
            if (g >= 0 && lane == __ffs(peers) - 1) head[g] = v;
            if (on) next2[2 * v] = above ? v + __ffs(above) : old;
            __syncwarp();
        }
    }
}

constexpr int kPer = kTinyNodes / kTopThreads;  // nodes per thread

// np: n rounded up to a multiple of 32; table null: preorder, depth and size only
__global__ void __launch_bounds__(kTopThreads)
    k_tiny_tree(const int32_t *__restrict__ parent, int n, int np, int32_t *__restrict__ pre,
                int32_t *__restrict__ depth, int32_t *__restrict__ size, int32_t *__restrict__ order,
                int32_t *__restrict__ table, int tlevels, int4 *__restrict__ nrec, int32_t *__restrict__ status) {
    pdl_prologue();
    extern __shared__ int32_t sm[];
    __shared__ TopShared sh;
    __shared__ int roots, root, bad;
    // a: first the next siblings, of node v in word 2 v; then the brackets' weights
    int32_t *par = sm, *head = sm + np, *nx = sm + 2 * np, *a = sm + 4 * np, *top = sm + 6 * np;
    const int tid = threadIdx.x;
    if (tid == 0) roots = root = bad = 0;
    __syncthreads();
    for (int v = tid; v < n; v += kTopThreads) {
        int32_t p = parent[v];
        if (p == -1) {
            atomicAdd(&roots, 1);
            root = v;
        } else if (p < 0 || p >= n) {
            bad = ETL_EBADTREE;
            p = -2;
        } else if (p == v) {
            bad = ETL_EBADTREE;
        }
        par[v] = p;
        head[v] = -1;
    }
    __syncthreads();
    // Children onto their parents' lists, in any order; then every node looks through its family's list for its
    // next sibling, the least larger label, and the least of all is the first child (a random tree of 1000
    // nodes 1 us, 9 by link_descending). In wide families all lanes walk the same list, a step at a time, while the
    // matching gets cheaper: 4096 nodes in families of 100 34 us all in all (37), of 250 55 (37).
    int32_t *some = nx, *link = nx + np;  // heads and links of the unordered lists; sizes in the odd words of a
    for (int v = tid; v < n; v += kTopThreads) {
        some[v] = -1;
        a[2 * v + 1] = 0;
    }
    __syncthreads();
    bool large = false;
    for (int v = tid; v < n; v += kTopThreads) {
        const int32_t p = par[v];
        if (p < 0) continue;
        link[v] = atomicExch(some + p, v);
        large |= atomicAdd(a + 2 * p + 1, 1) >= kFamily;
    }
    if (__syncthreads_or(large)) {
        if (tid < kWarp) link_descending(par, n, head, a);
    } else {
        for (int v = tid; v < n; v += kTopThreads) {
            const int32_t p = par[v];
            int32_t after = INT_MAX, least = INT_MAX;
            for (int32_t c = p >= 0 ? some[p] : -1; c >= 0; c = link[c]) {
                least = min(least, c);
                if (c > v) after = min(after, c);
            }
            a[2 * v] = after < INT_MAX ? after : -1;
            if (least == v) head[p] = v;
        }
    }
    __syncthreads();
    // the tour's list, leaves contracted (lca.cu): 2v enters v, 2v + 1 leaves it. A weight counts brackets in
    // its upper half and opening ones in its lower
    for (int v = tid; v < n; v += kTopThreads) {
        const int32_t p = par[v], h = head[v], x = a[2 * v];
        const int32_t c = x >= 0 ? 2 * x : p >= 0 ? 2 * p + 1 : kEndT;
        const bool leaf = h < 0 && p >= 0;
        nx[2 * v] = leaf ? c : h >= 0 ? 2 * h : 2 * v + 1;
        nx[2 * v + 1] = leaf ? kEndT : c;
        a[2 * v] = leaf ? 0x20001 : 0x10001;
        a[2 * v + 1] = 0x10000;
    }
    __syncthreads();
    rank_in_shared<false>(2 * n, 2 * root, (2 * n) << 16 | n, sh, nx, a, nullptr, &bad);
    int32_t pv[kPer], sv[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int v = tid + j * kTopThreads;
        pv[j] = sv[j] = -1;
        if (v >= n) continue;
        const bool leaf = head[v] < 0 && par[v] >= 0;
        const int32_t zo = nx[2 * v], zc = leaf ? zo : nx[2 * v + 1];
        int32_t d = -1;
        if (zo >= 0 || zc >= 0) {
            bad = ETL_EBADTREE;  // not on the list from the root
        } else {
            const int so = zo & ~kVisited, sc = zc & ~kVisited;
            const uint32_t at = uint32_t(sh.V1[so] + a[2 * v]);
            const int32_t r0 = int32_t(at >> 16), r1 = leaf ? r0 + 1 : int32_t(uint32_t(sh.V1[sc] + a[2 * v + 1]) >> 16);
            pv[j] = int32_t(at & 0xffff);
            sv[j] = (r1 - r0 + 1) >> 1;
            d = 2 * pv[j] - r0;
        }
        pre[v] = pv[j];
        depth[v] = d;
        size[v] = sv[j];
    }
    __syncthreads();
    int32_t *spre = head, *sorder = nx, *ssize = nx + np, *pm = a, *smin = a + np;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int v = tid + j * kTopThreads;
        if (v >= n) continue;
        spre[v] = pv[j];
        ssize[v] = sv[j];
        if (pv[j] >= 0 && pv[j] < n) {
            sorder[pv[j]] = v;
            order[pv[j]] = v;
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (roots != 1 || spre[root] != 0 || ssize[root] != n) bad = ETL_EBADTREE;
        *status = bad;
    }
    if (!table) return;
    // Q in preorder, prefix and suffix minima of its blocks of 32
    const int lane = tid & 31, nblk = np / kRmqBlock;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = tid + j * kTopThreads;
        if (i - lane >= np) continue;  // np is a multiple of 32: whole warps
        int32_t q = INT_MAX;
        if (i < n) {
            const int32_t v = sorder[i], p = v >= 0 && v < n ? par[v] : -1;
            q = p >= 0 ? spre[p] : -1;
        }
        int32_t a = q, b = q;
#pragma unroll
        for (int d = 1; d < kRmqBlock; d <<= 1) {
            const int32_t up = __shfl_up_sync(kFull, a, d), dn = __shfl_down_sync(kFull, b, d);
            if (lane >= d) a = min(a, up);
            if (lane + d < kRmqBlock) b = min(b, dn);
        }
        table[i] = q;
        reinterpret_cast<int2 *>(table + np)[i] = make_int2(a, b);
        pm[i] = a;
        smin[i] = b;
        if (lane == 31) {
            top[i >> kRmqBlockLog2] = a;
            table[3 * np + (i >> kRmqBlockLog2)] = a;
        }
    }
    __syncthreads();
    for (int l = 1; l < tlevels; ++l) {
        const int h = 1 << (l - 1);
        int32_t x = INT_MAX;
        if (tid < nblk) x = min(top[tid], tid + h < nblk ? top[tid + h] : INT_MAX);
        __syncthreads();
        if (tid < nblk) {
            top[tid] = x;
            table[3 * np + l * nblk + tid] = x;
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int v = tid + j * kTopThreads;
        if (v >= n) continue;
        const int32_t p = pv[j];
        nrec[v] = p >= 0 && p < n ? make_int4(p, pm[p], smin[p], sv[j]) : make_int4(p, INT_MAX, INT_MAX, sv[j]);
    }
}

size_t tiny_smem(int np) { return size_t(6 * np + np / kRmqBlock) * sizeof(int32_t); }

}  // namespace

etl_status build_tiny_tree(const int32_t *parent, etl_lca_s *h, cudaStream_t s) {
    const int n = h->n, np = int(h->bl.nblk) * kRmqBlock;
    cudaFuncSetAttribute(k_tiny_tree, cudaFuncAttributeMaxDynamicSharedMemorySize, int(tiny_smem(kTinyNodes)));
    PhaseTimer pt("lca.tiny", s);
    launch(k_tiny_tree, 1, kTopThreads, tiny_smem(np), s, parent, n, np, h->pre, h->depth, h->size, h->order,
           h->has_table ? h->table : nullptr, h->bl.tlevels, static_cast<int4 *>(h->nrec), h->status);
    note_launch();
    return last_launch();
}

}  // namespace etl
