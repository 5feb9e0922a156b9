// The list that the kNN selection (sj_knn.cu) ranks neighbours in, one warp's.
// The functions without a barrier also compile for the host, lane by lane.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace sj {

constexpr int kKnnList = 256;  // list entries of a warp (4 KB)
// Rank of a lane's place past the end of the list: above every k, so that such
// a lane writes nothing (a k above kKnnList pads the row behind the list's
// entries, and another lane writes that padding).
constexpr int kKnnPast = 0x7FFFFFFF;

struct KnnKey {
    uint32_t i, lo, hi;  // index, low and high half of the distance's bits
};
__host__ __device__ __forceinline__ KnnKey knn_key(int4 e) { return {(uint32_t)e.z, (uint32_t)e.x, (uint32_t)e.y}; }

// r - 1 when a < b, else r.
__host__ __device__ __forceinline__ int knn_minus_lt(int r, KnnKey a, KnnKey b) {
#ifdef __CUDA_ARCH__
    asm("{\n.reg .u32 t;\nsub.cc.u32 t, %1, %4;\nsubc.cc.u32 t, %2, %5;\nsubc.cc.u32 t, %3, %6;\n"
        "subc.u32 %0, %0, 0;\n}"
        : "+r"(r)
        : "r"(a.i), "r"(a.lo), "r"(a.hi), "r"(b.i), "r"(b.lo), "r"(b.hi));
    return r;
#else
    const uint64_t x = (uint64_t)a.hi << 32 | a.lo, y = (uint64_t)b.hi << 32 | b.lo;
    return x < y || (x == y && a.i < b.i) ? r - 1 : r;
#endif
}

// The entries 32 u + lane (u < E) of a list of m <= 32 E entries and their
// ranks (kKnnPast past the end).
template <int E>
__host__ __device__ __forceinline__ void knn_rank(const int4* list, int m, int lane, int4 (&e)[E], int (&rank)[E]) {
    KnnKey key[E];
#pragma unroll
    for (int u = 0; u < E; ++u) {
        e[u] = list[32 * u + lane < m ? 32 * u + lane : m - 1];
        key[u] = knn_key(e[u]);
        rank[u] = 0;
    }
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
        const KnnKey o = knn_key(list[j]);
#pragma unroll
        for (int u = 0; u < E; ++u) rank[u] = knn_minus_lt(rank[u], o, key[u]);
    }
#pragma unroll
    for (int u = 0; u < E; ++u) rank[u] = 32 * u + lane < m ? -rank[u] : kKnnPast;
}

// Cuts a list of m > k entries back to its k smallest, in order.
template <int E>
__device__ __forceinline__ void knn_cut(int4* list, int m, int k, int lane) {
    int4 e[E];
    int rank[E];
    knn_rank<E>(list, m, lane, e, rank);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (rank[u] < k) list[rank[u]] = e[u];
    __syncwarp();
}

// Writes the min(m, k) smallest of the list as row i of the outputs.
template <int E>
__host__ __device__ __forceinline__ void knn_write(const int4* list, int m, int k, int64_t i, int lane,
                                                   int32_t* idx_out, double* dist_out) {
    int4 e[E];
    int rank[E];
    knn_rank<E>(list, m, lane, e, rank);
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (rank[u] < k) {
            idx_out[i * k + rank[u]] = e[u].z;
            reinterpret_cast<int2*>(dist_out)[i * k + rank[u]] = make_int2(e[u].x, e[u].y);  // (the distance's bits)
        }
}

}  // namespace sj
