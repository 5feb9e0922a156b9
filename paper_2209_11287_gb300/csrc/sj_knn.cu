// The distance tile as a standalone operation, and k nearest neighbours
// from a join's result.
//
// sj_sqdist_tile: every squared distance between two point sets, the
// brute-force tile of the paper's Fig. 3 experiment (Sec. IV), in the
// decision rule's own arithmetic (binary64, dimension order, subtraction,
// product and sum each rounded, no contraction), so each value is exactly
// the s the join decides with.
//
// sj_knn_from_join: the k nearest of every point's eps-neighbours (the
// reuse of the join for kNN the paper names as future work, Sec. V): the
// pairs of a result with distances are bucketed by their first point and
// each bucket's k smallest (distance, index) are selected.
#include <algorithm>

#include "sj_internal.cuh"
#include "sj_knn_list.cuh"

namespace sj {

namespace {

constexpr int kTileQ = 64;  // rows of A per block
constexpr int kTileC = 64;  // rows of B per block
constexpr int kDimChunk = 16;

// One 64 x 64 output tile per block of 256 threads (4 x 4 values each); A
// and B rows staged in shared memory 16 dims at a time.
__global__ void __launch_bounds__(256) k_sqdist_tile(const double* __restrict__ A, int64_t m,
                                                     const double* __restrict__ B, int64_t nb, int d, double* out) {
    __shared__ double sa[kDimChunk][kTileQ + 1];
    __shared__ double sb[kDimChunk][kTileC + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t i0 = (int64_t)blockIdx.y * kTileQ, j0 = (int64_t)blockIdx.x * kTileC;
    double acc[4][4] = {};
    for (int k0 = 0; k0 < d; k0 += kDimChunk) {
        const int kc = min(kDimChunk, d - k0);
        for (int e = threadIdx.x; e < kDimChunk * kTileQ; e += 256) {
            const int r = e / kDimChunk, k = e % kDimChunk;
            const int64_t ia = i0 + r, jb = j0 + r;
            sa[k][r] = (k < kc && ia < m) ? A[ia * d + k0 + k] : 0.0;
            sb[k][r] = (k < kc && jb < nb) ? B[jb * d + k0 + k] : 0.0;
        }
        __syncthreads();
        for (int k = 0; k < kc; ++k) {  // dimension order, each operation rounded
            double a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = sa[k][ty + 16 * u];
                b[u] = sb[k][tx + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const double t = __dsub_rn(a[u], b[v]);
                    acc[u][v] = __dadd_rn(acc[u][v], __dmul_rn(t, t));
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
            if (i < m && j < nb) out[i * nb + j] = acc[u][v];
        }
}

// One neighbour of a bucket: 16 bytes, so a pair is one scattered store (one
// L2 sector) instead of two, and one load in the selection.
struct __align__(16) KnnEntry {
    double dist;
    int32_t idx;
    int32_t pad;
};

// kNN from a join: bucket sizes (self pairs left out) and every pair's place
// in its bucket, so the bucketing below needs no second atomic per pair (9.4 M
// pairs, both kernels: 213 us with an atomic in each and two stores per pair,
// 185 us so) ...  These take 20 bytes a pair; where that finds no room, or
// where it is far more than L2 holds and the buckets are long (knn_split), the
// entries are split (12 bytes a pair: no place, one atomic more).
template <bool PLACE>
__global__ void k_knn_degree(const int2* __restrict__ pairs, long long count, uint32_t* deg,
                             uint32_t* __restrict__ place) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < count;
         p += (long long)gridDim.x * blockDim.x) {
        const int2 e = pairs[p];
        if (e.x == e.y) continue;
        if constexpr (PLACE)
            place[p] = atomicAdd(&deg[e.x], 1u);
        else
            atomicAdd(&deg[e.x], 1u);
    }
}

// ... the pairs bucketed by their first point ...
__global__ void k_knn_bucket(const int2* __restrict__ pairs, const double* __restrict__ dist, long long count,
                             const uint32_t* __restrict__ off, const uint32_t* __restrict__ place, KnnEntry* nb) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < count;
         p += (long long)gridDim.x * blockDim.x) {
        const int2 e = pairs[p];
        if (e.x == e.y) continue;
        const long long d = __double_as_longlong(dist[p]);
        *reinterpret_cast<int4*>(nb + off[e.x] + place[p]) = make_int4((int)d, (int)(d >> 32), e.y, 0);
    }
}

__global__ void k_knn_bucket_split(const int2* __restrict__ pairs, const double* __restrict__ dist, long long count,
                                   const uint32_t* __restrict__ off, uint32_t* cursor, int32_t* nb_idx,
                                   double* nb_dist) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < count;
         p += (long long)gridDim.x * blockDim.x) {
        const int2 e = pairs[p];
        if (e.x == e.y) continue;
        const uint32_t s = off[e.x] + atomicAdd(&cursor[e.x], 1u);
        nb_idx[s] = e.y;
        nb_dist[s] = dist[p];
    }
}

// Long buckets beyond L2 fill their lines before they are evicted only if few of
// them are open at a time: then the fewer bytes of the split entries count for
// more than the second atomic, most of all where the pairs of a point lie
// scattered in the list (a tensor-core filter's).  The whole call at k = 8, whole
// / split, us: 30,000 points x 1,700 neighbours 16-D clusters 2295 / 1696, 1,780
// uniform 16-D 2522 / 1867, 1,370 3-D 1494 / 1468; 100,000 x 770 16-D 3873 / 2942,
// x 640 3-D 2238 / 1983, x 300 16-D clusters 1407 / 1241, x 285 3-D 1013 / 974, x
// 146 541 / 527; 30,000 x 630 706 / 727; shorter or fewer: 1,000,000 x 41 1849 /
// 1919, 30,000 x 360 432 / 460.
static bool knn_split(long long count, int64_t n) { return count >= (3 << 22) && count / n >= 128; }

// Where the selection reads its entries (as KnnEntry's four words), and whether
// it loads a chunk ahead, so that the load does not wait for the list: it pays for
// long buckets (150 neighbours of 100,000 points 502 / 488 us), not for short ones
// (47 neighbours 150 / 160).
struct KnnWhole {
    static constexpr bool kAhead = false;
    const int4* e;
    __device__ __forceinline__ int4 operator[](uint32_t s) const { return __ldg(e + s); }
};
struct KnnSplit {
    static constexpr bool kAhead = true;
    const int32_t* idx;
    const double* dist;
    __device__ __forceinline__ int4 operator[](uint32_t s) const {
        const long long d = __double_as_longlong(dist[s]);
        return make_int4((int)d, (int)(d >> 32), idx[s], 0);
    }
};

// ... and, one warp per point, its k smallest by (distance, index).
//
// The warp gathers candidates in a list of kKnnList entries in shared memory
// and ranks them there: an entry's rank is the number of list entries below
// it, counted by every lane for its own entries against each entry in turn
// (a shared-memory broadcast).  A distance is not negative, so its bits order
// as an integer, and (distance bits, index) compare as one 96-bit integer: a
// borrow chain of four 32-bit subtractions, no FP64 instruction (that pipe
// runs at 1/64 of the integer rate here) and no case for equal distances.  A
// bucket that fits the list is ranked once; a longer one is cut back to its k
// smallest whenever the list holds 2 k entries (at least 64), and from then on
// only entries below the k-th of those enter: ranking m entries costs m^2.  k
// rounds of a warp-wide minimum over the whole bucket, the earlier form, took a
// pass over the bucket and ten shuffles per neighbour; it remains for k above
// kKnnCut with longer buckets, which the list cannot hold.  Bound by
// instruction issue (four instructions per pair of entries and lane).
// Measured, rounds / list: 200,003 points, 47 neighbours, k = 16: 3424 / 150
// us; 200,000 points, 57 neighbours, k = 8: 1798 / 149 us; 100,000 16-D points,
// 50 neighbours on average, k = 32: 2943 / 166 us (cut back at the full list
// only: 299).
constexpr int kKnnCut = kKnnList - 64;   // largest k the list is cut back to
// Up to this k the first 32 neighbours are cut back at once: the k-th of them
// keeps most of the rest out, and the final ranking is over about
// k + (bucket - 32) k / 32 entries (47 neighbours, k = 16: 209 us without, 150
// us with; the two rankings cost more than the one from about 3/4 of 32 on).
constexpr int kKnnEarly = 24;
constexpr int kKnnWarps = 8;

template <typename Src>
__global__ void __launch_bounds__(32 * kKnnWarps) k_knn_select(int64_t n, int k, const uint32_t* __restrict__ off,
                                                               const Src src, int32_t* idx_out, double* dist_out,
                                                               int32_t* found_out) {
    __shared__ int4 s_list[kKnnWarps][kKnnList];
    const int lane = threadIdx.x & 31;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const uint32_t a = off[i], b = off[i + 1];
    const int found = (int)min(b - a, (uint32_t)k);
    if (b - a <= (uint32_t)kKnnList || k <= kKnnCut) {
        int4* list = s_list[threadIdx.x >> 5];
        const int full = min(kKnnList - 31, max(64, 2 * k));  // cut back from this many on
        int m = 0;
        KnnKey bar{0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};  // the k-th smallest so far
        int4 next = make_int4(0, 0, 0, 0);
        if (Src::kAhead && a + (uint32_t)lane < b) next = src[a + (uint32_t)lane];
        for (uint32_t s0 = a; s0 < b; s0 += 32) {
            const uint32_t s = s0 + (uint32_t)lane;
            int4 e = next;
            if constexpr (Src::kAhead) {
                if (b - s0 > 32u + (uint32_t)lane) next = src[s + 32u];
            } else if (s < b) {
                e = src[s];
            }
            const bool in = s < b && knn_minus_lt(0, knn_key(e), bar) != 0;
            const unsigned w = __ballot_sync(0xffffffffu, in);
            if (in) list[m + __popc(w & ((1u << lane) - 1u))] = e;
            m += __popc(w);
            __syncwarp();
            // (a list this full holds more than k entries, and room for 32)
            if (b - s0 > 32u && (m >= full || (s0 == a && k <= kKnnEarly))) {
                if (m <= 32)
                    knn_cut<1>(list, m, k, lane);
                else if (m <= 64)
                    knn_cut<2>(list, m, k, lane);
                else if (m <= 128)
                    knn_cut<4>(list, m, k, lane);
                else
                    knn_cut<kKnnList / 32>(list, m, k, lane);
                m = k;
                bar = knn_key(list[k - 1]);
            }
        }
        if (m > 0) {
            if (m <= 32)
                knn_write<1>(list, m, k, i, lane, idx_out, dist_out);
            else if (m <= 64)
                knn_write<2>(list, m, k, i, lane, idx_out, dist_out);
            else if (m <= 128)
                knn_write<4>(list, m, k, i, lane, idx_out, dist_out);
            else
                knn_write<kKnnList / 32>(list, m, k, i, lane, idx_out, dist_out);
        }
    } else {
        // k rounds of a warp-wide minimum above the last one taken
        KnnKey last{0, 0, 0};
        for (int r = 0; r < found; ++r) {
            KnnKey best{0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
            for (uint32_t s = a + lane; s < b; s += 32) {
                const KnnKey e = knn_key(src[s]);
                if ((r == 0 || knn_minus_lt(0, last, e)) && knn_minus_lt(0, e, best)) best = e;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                KnnKey x;
                x.i = __shfl_xor_sync(0xffffffffu, best.i, o);
                x.lo = __shfl_xor_sync(0xffffffffu, best.lo, o);
                x.hi = __shfl_xor_sync(0xffffffffu, best.hi, o);
                if (knn_minus_lt(0, x, best)) best = x;
            }
            if (lane == 0) {
                idx_out[i * k + r] = (int32_t)best.i;
                dist_out[i * k + r] = __hiloint2double((int)best.hi, (int)best.lo);
            }
            last = best;
        }
    }
    for (int r = found + lane; r < k; r += 32) {
        idx_out[i * k + r] = -1;
        dist_out[i * k + r] = INFINITY;
    }
    if (lane == 0) found_out[i] = found;
}

unsigned grid_for(long long work, int device) {
    const long long cap = (long long)device_sm_count(device) * 16;
    long long b = (work + 255) / 256;
    return (unsigned)std::max<long long>(1, std::min(b, cap));
}

}  // namespace

}  // namespace sj

using namespace sj;

extern "C" int sj_sqdist_tile(const double* A, int64_t m, const double* B, int64_t nb, int32_t d, double* out,
                              void* stream) {
    clear_error();
    if (!A || !B || !out || m < 1 || nb < 1 || d < 1 || d > SJ_MAX_D || m > 0x7FFFFFFFll || nb > 0x7FFFFFFFll) {
        set_error("invalid argument");
        return SJ_ERR_ARG;
    }
    if (!is_device_pointer(A) || !is_device_pointer(B) || !is_device_pointer(out)) {
        set_error("sj_sqdist_tile needs device pointers");
        return SJ_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const dim3 grid((unsigned)((nb + kTileC - 1) / kTileC), (unsigned)((m + kTileQ - 1) / kTileQ));
    if (grid.y > 65535u) {
        set_error("m = %lld rows of A exceed one launch (at most %lld)", (long long)m, 65535ll * kTileQ);
        return SJ_ERR_ARG;
    }
    k_sqdist_tile<<<grid, 256, 0, s>>>(A, m, B, nb, d, out);
    note_launch();
    SJ_CK(cudaGetLastError());
    return SJ_OK;
}

extern "C" int sj_knn_from_join(const sj_result* r, int64_t n, int32_t k, int32_t* idx_out, double* dist_out,
                                int32_t* found_out) {
    clear_error();
    if (!r || !idx_out || !dist_out || !found_out || n < 1 || n > 0x7FFFFFFFll || k < 1 || k > 1024) {
        set_error("invalid argument");
        return SJ_ERR_ARG;
    }
    const ResultImpl* ri = static_cast<const ResultImpl*>(r->internal);
    if (r->count > 0 && (!ri || !ri->block || ri->shared_pool)) {
        set_error("sj_knn_from_join takes the result of a single join (sj_self_join / sj_join)");
        return SJ_ERR_ARG;
    }
    if (r->count > 0 && (!r->has_distances || !ri->dblock)) {
        set_error("sj_knn_from_join needs a result with distances (sj_options.emit_distances = 1)");
        return SJ_ERR_ARG;
    }
    if (r->count > (int64_t)r->n_pages * r->page_pairs) {
        set_error("the result holds only part of its pairs");
        return SJ_ERR_RESULT_OVERFLOW;
    }
    cudaStream_t s = ri ? ri->stream : nullptr;
    int dev = 0;
    SJ_CK(cudaGetDevice(&dev));
    const long long count = (long long)r->count;
    const int2* pairs = ri ? reinterpret_cast<const int2*>(ri->block) : nullptr;
    const double* dist = ri ? ri->dblock : nullptr;
    Scratch tmp(s);
    int32_t *oi = nullptr, *of = nullptr;
    uint32_t *deg = nullptr, *off = nullptr, *place = nullptr;
    KnnEntry* nb = nullptr;
    int32_t* nb_idx = nullptr;
    double *nb_dist = nullptr, *od = nullptr;
    const size_t slots = (size_t)std::max<long long>(count, 1);
    SJ_TRY(tmp.alloc(&deg, (size_t)n));
    SJ_TRY(tmp.alloc(&off, (size_t)n + 1));
    SJ_TRY(tmp.alloc(&oi, (size_t)n * k));
    SJ_TRY(tmp.alloc(&od, (size_t)n * k));
    SJ_TRY(tmp.alloc(&of, (size_t)n));
    int st = knn_split(count, n) ? SJ_ERR_OOM : dev_alloc_t(&nb, slots, s);
    if (st == SJ_OK) st = dev_alloc_t(&place, slots, s);
    if (st == SJ_ERR_OOM) {  // the split entries then
        clear_error();
        dev_free(nb, s);
        nb = nullptr;
        SJ_TRY(tmp.alloc(&nb_idx, slots));
        SJ_TRY(tmp.alloc(&nb_dist, slots));
    } else if (st != SJ_OK) {
        dev_free(nb, s);
        return st;
    } else {
        tmp.ptrs.push_back(nb);
        tmp.ptrs.push_back(place);
    }
    SJ_CK(cudaMemsetAsync(deg, 0, (size_t)n * sizeof(uint32_t), s));
    if (count > 0) {
        if (place)
            k_knn_degree<true><<<grid_for(count, dev), 256, 0, s>>>(pairs, count, deg, place);
        else
            k_knn_degree<false><<<grid_for(count, dev), 256, 0, s>>>(pairs, count, deg, nullptr);
        note_launch();
        SJ_CK(cudaGetLastError());
    }
    SJ_TRY(scan_exclusive_u32_total(deg, off, n, s));  // off[n]: the total
    if (count > 0) {
        if (nb) {
            k_knn_bucket<<<grid_for(count, dev), 256, 0, s>>>(pairs, dist, count, off, place, nb);
        } else {
            SJ_CK(cudaMemsetAsync(deg, 0, (size_t)n * sizeof(uint32_t), s));  // the buckets' cursors
            k_knn_bucket_split<<<grid_for(count, dev), 256, 0, s>>>(pairs, dist, count, off, deg, nb_idx, nb_dist);
        }
        note_launch();
        SJ_CK(cudaGetLastError());
    }
    const unsigned gs = (unsigned)((n + kKnnWarps - 1) / kKnnWarps);
    if (nb)
        k_knn_select<<<gs, 32 * kKnnWarps, 0, s>>>(n, k, off, KnnWhole{reinterpret_cast<const int4*>(nb)}, oi, od, of);
    else
        k_knn_select<<<gs, 32 * kKnnWarps, 0, s>>>(n, k, off, KnnSplit{nb_idx, nb_dist}, oi, od, of);
    note_launch();
    SJ_CK(cudaGetLastError());
    SJ_CK(cudaMemcpyAsync(idx_out, oi, (size_t)n * k * sizeof(int32_t), cudaMemcpyDefault, s));
    SJ_CK(cudaMemcpyAsync(dist_out, od, (size_t)n * k * sizeof(double), cudaMemcpyDefault, s));
    SJ_CK(cudaMemcpyAsync(found_out, of, (size_t)n * sizeof(int32_t), cudaMemcpyDefault, s));
    SJ_CK(cudaStreamSynchronize(s));
    return SJ_OK;
}
