// DBSCAN on the result of a self-join: the join's eps-neighbourhoods reused
// for density-based clustering (the paper names this reuse of its join as
// future work, Sec. V).
//
// Definition (Ester et al. 1996, on the neighbourhoods the join returns): a
// point is core iff its neighbourhood, itself included, holds at least
// min_pts points; clusters are the connected components of the core points
// under the core-core pairs; a non-core point with a core neighbour is a
// border point and joins the smallest of its core neighbours' clusters; the
// rest is noise (-1).  Clusters are numbered by their smallest core point.
//
// Components come from a lock-free union-find over the core-core pairs:
// roots are always hooked under the smaller root (parent[x] <= x holds at
// every moment, so every find terminates and a component's root is its
// smallest core point), finds halve their paths, a failed hook retries.
//
// Walking the forest twice for every pair is a chain of dependent loads, and
// almost all of these walks only find that the points are united already
// (2M 4-D points, 121M pairs: 6163 us of the 7080 us after the join).  So a few
// rounds on a share of the pairs first join nearly everything without a walk
// (k_db_hook, the forest flattened after each), and the pass over all pairs
// compares two cached ancestors and walks for the rest only, 32 at a time
// (the rounds with their flattenings 280 us, the pass 270).  What is left are three reads of the pair
// list (0.97 GB, 143 us each at the copy rate) and the lookups that go with
// them: k_db_degree 641 -> 337 us (one atomic per distinct point of a warp),
// k_db_border 388 -> 257 us (core points as a bit set, four pairs a lane in
// flight).
#include <algorithm>

#include "sj_internal.cuh"

namespace sj {

namespace {

constexpr int32_t kNoLabel = 0x7FFFFFFF;
constexpr int kUnionTries = 1 << 20;  // retries of one union (each failure is another thread's progress)

// Passes over the pairs: a warp takes kDbAhead of every `stride`-th block of
// 32 pairs at a time (from block `first` on; (-1, -1) past the end), so that
// each step of a pass has that many independent loads of a lane in flight.
constexpr int kDbAhead = 4;
constexpr int kDbThreads = 256;
struct DbPairs {
    const int2* pairs;
    long long count, block, step;  // pairs, the warp's next block, blocks between its loads
    __device__ DbPairs(const int2* p, long long n, int stride, int first) : pairs(p), count(n) {
        const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
        block = warp * stride + first;
        step = (long long)gridDim.x * (blockDim.x >> 5) * stride;
    }
    __device__ __forceinline__ bool next(int2 (&e)[kDbAhead]) {
        if (block * 32 >= count) return false;
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            const long long p = (block + u * step) * 32 + (threadIdx.x & 31);
            e[u] = p < count ? pairs[p] : make_int2(-1, -1);
        }
        block += kDbAhead * step;
        return true;
    }
};

// Neighbourhood sizes.  Neighbouring pairs of a join share their points (a
// work item's queries, a candidate's copies), so the lanes of a warp with the
// same first point add with one atomic.
__global__ void __launch_bounds__(kDbThreads) k_db_degree(const int2* __restrict__ pairs, long long count,
                                                          int32_t* deg) {
    const int lane = threadIdx.x & 31;
    DbPairs in(pairs, count, 1, 0);
    int2 e[kDbAhead];
    while (in.next(e)) {
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            const unsigned same = __match_any_sync(0xffffffffu, e[u].x);
            if (e[u].x >= 0 && lane == __ffs(same) - 1) atomicAdd(&deg[e[u].x], __popc(same));
        }
    }
}

// Core points as a bit set (small enough to stay in L1 where the pair passes
// test it), and whether there are others.
__global__ void k_db_core(int64_t n, const int32_t* __restrict__ deg, int32_t min_pts, uint32_t* core,
                          unsigned long long* others) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool c = i < n && deg[i] >= min_pts;
    const unsigned w = __ballot_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && i < n) core[i >> 5] = w;
    const int o = __syncthreads_or(i < n && !c);
    if (threadIdx.x == 0 && o) *others = 1;  // (every writer writes the same)
}

__device__ __forceinline__ bool db_core(const uint32_t* __restrict__ core, int32_t i) {
    return (core[i >> 5] >> (i & 31)) & 1u;
}

// The core-core pairs of e, each once (first point below the second).
__device__ __forceinline__ void db_core_pairs(const int2 (&e)[kDbAhead], const uint32_t* __restrict__ core,
                                              bool (&take)[kDbAhead]) {
    uint32_t cx[kDbAhead], cy[kDbAhead];
#pragma unroll
    for (int u = 0; u < kDbAhead; ++u) {
        take[u] = e[u].x < e[u].y;  // ((-1, -1) is left out too)
        cx[u] = take[u] ? core[e[u].x >> 5] : 0u;
        cy[u] = take[u] ? core[e[u].y >> 5] : 0u;
    }
#pragma unroll
    for (int u = 0; u < kDbAhead; ++u) take[u] = ((cx[u] >> (e[u].x & 31)) & (cy[u] >> (e[u].y & 31)) & 1u) != 0u;
}

// (`status`: the error flag and the flag of k_db_core)
__global__ void k_db_init(int64_t n, int32_t* parent, int32_t* border, int32_t* deg, unsigned long long* status) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        parent[i] = (int32_t)i;
        border[i] = kNoLabel;
        deg[i] = 0;
    }
    if (i < 2) status[i] = 0;  // (n >= 1: at least one whole block)
}

__device__ __forceinline__ int32_t db_find(volatile int32_t* parent, int32_t x) {
    for (;;) {  // indices strictly decrease along the path: this ends
        const int32_t p = parent[x];
        if (p == x) return x;
        const int32_t gp = parent[p];
        if (gp != p) parent[x] = gp;  // path halving (x is not a root)
        x = p;
    }
}

// A round of hooking on a share of the pairs: where the two points have
// different roots (the forest is flat), the larger root goes under the
// smaller.  No walk and no retry: a hook that another one replaces is only
// lost time, k_db_union sees every pair.
__global__ void __launch_bounds__(kDbThreads) k_db_hook(const int2* __restrict__ pairs, long long count, int stride,
                                                        int first, const uint32_t* __restrict__ core,
                                                        const int32_t* root, int32_t* parent) {
    DbPairs in(pairs, count, stride, first);
    int2 e[kDbAhead];
    while (in.next(e)) {
        bool take[kDbAhead];
        db_core_pairs(e, core, take);
        int32_t a[kDbAhead], b[kDbAhead];
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            a[u] = take[u] ? root[e[u].x] : 0;
            b[u] = take[u] ? root[e[u].y] : 0;
        }
        int32_t now[kDbAhead];  // (a look first: late rounds hook few roots from many pairs)
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) now[u] = a[u] != b[u] ? __ldcg(&parent[max(a[u], b[u])]) : 0;
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u)
            if (a[u] != b[u] && min(a[u], b[u]) < now[u]) atomicMin(&parent[max(a[u], b[u])], min(a[u], b[u]));
    }
}

// Unites two points (bounded retries; each failure is another thread's
// progress).
__device__ __forceinline__ void db_unite(int2 e, int32_t* parent, unsigned long long* error) {
    volatile int32_t* par = parent;
    for (int tries = 0;; ++tries) {
        if (tries == kUnionTries) {
            atomicExch(error, 1ull);
            break;
        }
        int32_t a = db_find(par, e.x), b = db_find(par, e.y);
        if (a == b) break;
        if (a > b) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(&parent[b], b, a) == b) break;  // the larger root under the smaller
    }
}

// Unites all core-core pairs.  `hint` is the forest read without regard to
// the writes going on: two points with the same ancestor there are in one set
// for good, and after the hooking rounds almost every pair is seen to be so
// from these two cached loads.  The others are queued, and the warp walks the
// forest for 32 of them at a time.
__global__ void __launch_bounds__(kDbThreads) k_db_union(const int2* __restrict__ pairs, long long count,
                                                         const uint32_t* __restrict__ core, const int32_t* hint,
                                                         int32_t* parent, unsigned long long* error) {
    __shared__ int2 s_queue[kDbThreads / 32][64];
    int2* queue = s_queue[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    int queued = 0;
    DbPairs in(pairs, count, 1, 0);
    int2 e[kDbAhead];
    while (in.next(e)) {
        bool take[kDbAhead];
        db_core_pairs(e, core, take);
        int32_t a[kDbAhead], b[kDbAhead];
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            a[u] = take[u] ? hint[e[u].x] : 0;
            b[u] = take[u] ? hint[e[u].y] : 0;
        }
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            const unsigned w = __ballot_sync(0xffffffffu, a[u] != b[u]);
            if (a[u] != b[u]) queue[queued + __popc(w & ((1u << lane) - 1u))] = e[u];
            queued += __popc(w);
            if (queued >= 32) {
                queued -= 32;
                __syncwarp();
                db_unite(queue[queued + lane], parent, error);
                __syncwarp();
            }
        }
    }
    __syncwarp();
    if (lane < queued) db_unite(queue[lane], parent, error);
}

// Every core point directly under its root, by pointer jumping.  A thread
// writes its own point's parent only: halving the paths of others here could
// put an older ancestor back over a root already stored.
__global__ void k_db_flatten(int64_t n, const uint32_t* __restrict__ core, int32_t* parent) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || !db_core(core, (int32_t)i)) return;
    volatile int32_t* par = parent;
    int32_t p = par[i];
    for (;;) {  // (ancestors only fall: this ends)
        const int32_t g = par[p];
        if (g == p) break;
        p = g;
        par[i] = p;
    }
}

// Border points: the smallest root among the core neighbours.
__global__ void __launch_bounds__(kDbThreads) k_db_border(const int2* __restrict__ pairs, long long count,
                                                          const uint32_t* __restrict__ core,
                                                          const unsigned long long* __restrict__ others,
                                                          const int32_t* __restrict__ parent, int32_t* border) {
    if (*others == 0) return;  // every point is core
    DbPairs in(pairs, count, 1, 0);
    int2 e[kDbAhead];
    while (in.next(e)) {
        uint32_t cx[kDbAhead], cy[kDbAhead];
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            const bool live = e[u].x >= 0;
            cx[u] = live ? core[e[u].x >> 5] : 0u;
            cy[u] = live ? core[e[u].y >> 5] : 0u;
        }
        int32_t r[kDbAhead], now[kDbAhead];
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u) {
            const bool take = (~(cx[u] >> (e[u].x & 31)) & (cy[u] >> (e[u].y & 31)) & 1u) != 0u;
            r[u] = take ? parent[e[u].y] : kNoLabel;
            now[u] = take ? border[e[u].x] : 0;  // (it only falls: a stale value costs an atomic)
        }
#pragma unroll
        for (int u = 0; u < kDbAhead; ++u)
            if (r[u] < now[u]) atomicMin(&border[e[u].x], r[u]);
    }
}

__global__ void k_db_roots(int64_t n, const uint32_t* __restrict__ core, const int32_t* __restrict__ parent,
                           uint32_t* flag) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) flag[i] = (db_core(core, (int32_t)i) && parent[i] == (int32_t)i) ? 1u : 0u;
}

__global__ void k_db_label(int64_t n, const uint32_t* __restrict__ core, const int32_t* __restrict__ parent,
                           const int32_t* __restrict__ border, const uint32_t* __restrict__ flag,
                           const uint32_t* __restrict__ rank, int32_t* labels, unsigned long long* clusters) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == n - 1) *clusters = (unsigned long long)rank[i] + flag[i];
    int32_t l = -1;
    if (db_core(core, (int32_t)i))
        l = (int32_t)rank[parent[i]];
    else if (border[i] != kNoLabel)
        l = (int32_t)rank[border[i]];
    labels[i] = l;
}

unsigned grid_for(long long work, int device) {
    const long long cap = (long long)device_sm_count(device) * 16;
    long long b = (work + 255) / 256;
    return (unsigned)std::max<long long>(1, std::min(b, cap));
}

// Hooking rounds, and the stride of their blocks of pairs: about kDbShare
// pairs a point each.  (Everything after the join, for 2M 4-D points with 121M
// pairs / 700,003 3-D points with 17M / 500,000 16-D points with 41M, by rounds
// and share, with path-halving flattenings: 3 x 6 1.55 / 0.61 / 0.85 ms, 2 x 6
// 1.80 / 0.60 / 0.82, 3 x 4 1.65 / 0.60 / 0.83, 3 x 2 1.77 / 0.74 / 0.85, 2 x 16
// 1.65 / 0.63 / 0.79.)
constexpr int kDbRounds = 3;
constexpr int kDbShare = 6;
int db_stride(long long count, int64_t n) {
    return (int)std::max<long long>(1, std::min<long long>(count / (n * kDbShare), 1 << 20));
}
// Few pairs of few neighbours go straight to the union pass, where the rounds'
// launches cost more than the walks (the whole call, with three read-backs
// instead of one about 25 us longer than now, us, 0 / 1 / 3 rounds, by points x
// neighbours, uniform 2-D to 4-D: 300 x 4 106 / 114 / 125, 3,000 x 4
// 123 / 129 / 134, 10,000 x 4 170 / 170 / 158, 300,000 x 4 577 / 753 / 319; from
// about 6 neighbours on three rounds are at least as fast at any size: 3,000 x
// 11 170 / 182 / 132, 100,000 x 10 781 / 739 / 245, 300 x 42 137 / 131 / 124).
int db_rounds(long long count, int64_t n) { return count < kDbShare * n && count < (1 << 15) ? 0 : kDbRounds; }

}  // namespace

}  // namespace sj

using namespace sj;

extern "C" int sj_dbscan(const sj_result* r, int64_t n, int32_t min_pts, int32_t* labels_out, int64_t* n_clusters) {
    clear_error();
    if (!r || !labels_out || n < 1 || n > 0x7FFFFFFFll || min_pts < 1) {
        set_error("invalid argument");
        return SJ_ERR_ARG;
    }
    const ResultImpl* ri = static_cast<const ResultImpl*>(r->internal);
    if (r->count > 0 && (!ri || !ri->block || ri->shared_pool)) {
        set_error("sj_dbscan takes the result of a single join (sj_self_join / sj_join)");
        return SJ_ERR_ARG;
    }
    if (r->count > (int64_t)r->n_pages * r->page_pairs) {
        set_error("the result holds %lld of its %lld pairs", (long long)r->n_pages * r->page_pairs,
                  (long long)r->count);
        return SJ_ERR_RESULT_OVERFLOW;
    }
    cudaStream_t s = ri ? ri->stream : nullptr;
    int dev = 0;
    SJ_CK(cudaGetDevice(&dev));
    const int2* pairs = ri ? reinterpret_cast<const int2*>(ri->block) : nullptr;
    const long long count = (long long)r->count;
    Scratch tmp(s);
    int32_t *deg = nullptr, *parent = nullptr, *border = nullptr, *labels = nullptr;
    uint32_t *flag = nullptr, *core = nullptr;  // flag: n flags, then n + 1 ranks
    unsigned long long* error = nullptr;        // the error flag; whether a point is not core, later the clusters
    SJ_TRY(tmp.alloc(&deg, (size_t)n));
    SJ_TRY(tmp.alloc(&parent, (size_t)n));
    SJ_TRY(tmp.alloc(&border, (size_t)n));
    SJ_TRY(tmp.alloc(&labels, (size_t)n));
    SJ_TRY(tmp.alloc(&flag, (size_t)2 * n + 1));
    SJ_TRY(tmp.alloc(&core, (size_t)((n + 31) / 32)));
    SJ_TRY(tmp.alloc(&error, 2));
    uint32_t* rank = flag + n;
    const unsigned gn = (unsigned)((n + 255) / 256);
    k_db_init<<<gn, 256, 0, s>>>(n, parent, border, deg, error);
    note_launch();
    if (count > 0) {
        k_db_degree<<<grid_for(count, dev), kDbThreads, 0, s>>>(pairs, count, deg);
        note_launch();
    }
    k_db_core<<<gn, 256, 0, s>>>(n, deg, min_pts, core, error + 1);
    note_launch();
    if (count > 0) {
        // hooking rounds on a share of the pairs each, then all of them
        const int stride = db_stride(count, n);
        const int rounds = db_rounds(count, n);
        for (int r = 0; r < rounds; ++r) {
            k_db_hook<<<grid_for(count / stride, dev), kDbThreads, 0, s>>>(
                pairs, count, stride, (int)((long long)r * stride / rounds), core, parent, parent);
            note_launch();
            k_db_flatten<<<gn, 256, 0, s>>>(n, core, parent);
            note_launch();
        }
        k_db_union<<<grid_for(count, dev), kDbThreads, 0, s>>>(pairs, count, core, parent, parent, error);
        note_launch();
        k_db_flatten<<<gn, 256, 0, s>>>(n, core, parent);
        note_launch();
        k_db_border<<<grid_for(count, dev), kDbThreads, 0, s>>>(pairs, count, core, error + 1, parent, border);
        note_launch();
    }
    k_db_roots<<<gn, 256, 0, s>>>(n, core, parent, flag);
    note_launch();
    SJ_CK(cudaGetLastError());
    SJ_TRY(scan_exclusive_u32(flag, rank, n, s));
    k_db_label<<<gn, 256, 0, s>>>(n, core, parent, border, flag, rank, labels, error + 1);
    note_launch();
    SJ_CK(cudaGetLastError());
    unsigned long long got[2] = {0, 0};  // the error flag, the number of clusters
    void* hs = host_staging(sizeof got);  // pinned: a direct copy
    SJ_CK(cudaMemcpyAsync(hs ? hs : got, error, sizeof got, cudaMemcpyDeviceToHost, s));
    SJ_CK(cudaMemcpyAsync(labels_out, labels, (size_t)n * sizeof(int32_t), cudaMemcpyDefault, s));
    SJ_CK(cudaStreamSynchronize(s));
    if (hs) memcpy(got, hs, sizeof got);
    if (got[0]) {
        set_error("a union-find update ran out of retries");
        return SJ_ERR_TIMEOUT;
    }
    if (n_clusters) *n_clusters = (int64_t)got[1];
    return SJ_OK;
}
