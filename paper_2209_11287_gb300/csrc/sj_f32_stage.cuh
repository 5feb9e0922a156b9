// Parts shared by the FP32 filters for small dimensions (sj_join_f32s.cu,
// sj_join_f32r.cu): candidate rows as vector loads and the warp's stage of
// pairs with a mirror flag.
#pragma once

#include "sj_join_common.cuh"

namespace sj {

// Candidate coordinates of one point as DP floats, loaded with vector loads.
template <int DP>
__device__ __forceinline__ void load_coords(const float* __restrict__ Y, int32_t j, float (&c)[DP]) {
    if constexpr (DP == 2) {
        const float2 v = reinterpret_cast<const float2*>(Y)[j];
        c[0] = v.x;
        c[1] = v.y;
    } else {
#pragma unroll
        for (int h = 0; h < DP / 4; ++h) {
            const float4 v = reinterpret_cast<const float4*>(Y)[(int64_t)j * (DP / 4) + h];
            c[4 * h] = v.x;
            c[4 * h + 1] = v.y;
            c[4 * h + 2] = v.z;
            c[4 * h + 3] = v.w;
        }
    }
}

// The warp's shared memory (W below) counts in `smir` the staged entries that
// are flagged for a mirrored copy (lane 0).
// Stage entries: (query output index | kStageMirror if the pair is also
// emitted mirrored, candidate output index); output indices are below 2^31.
constexpr uint32_t kStageMirror = 0x80000000u;

// Copies the warp's staged entries out: one atomic on the result cursor (the
// instance's cursor in a batched join) reserves entries + mirrored pairs;
// entry i goes to base + i, the mirrored pairs after them in entry order.
// Positions past the pool's capacity (a batched instance's pages) are counted
// but not written.
// BATCH: whether the pairs may belong to a batched join.
template <bool BATCH = true, typename W_t>
__device__ __forceinline__ void f32s_flush(W_t& W, WarpStage& st, const JoinParams& P, int lane) {
    __syncwarp();
    const int ne = st.cnt;
    const unsigned long long total = (unsigned long long)(ne + W.smir);
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long base = 0;
    if (BATCH && P.batch) {
        const BatchJoin& B = *P.batch;
        if (lane == 0 && total > 0) base = atomicAdd(&B.cursor[st.gid], total);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (total > 0) {
            // pages of at least 64 pairs: a flush of <= kStageMax pairs
            // touches at most 32 pages, one lane resolves each
            const unsigned long long pg0 = base >> B.page_log2;
            const int npg = (int)(((base + total - 1ull) >> B.page_log2) - pg0) + 1;
            const int32_t mine = lane < npg ? batch_page(B, st.gid, pg0 + (unsigned long long)lane) : -1;
            const unsigned long long mask = (1ull << B.page_log2) - 1ull;
            unsigned long long mb = base + (unsigned long long)ne;
            for (int i0 = 0; i0 < ne; i0 += 32) {
                const int i = i0 + lane;
                const int2 e = i < ne ? st.pairs[i] : make_int2(0, 0);
                const bool m = i < ne && ((uint32_t)e.x & kStageMirror) != 0u;
                const int32_t qi = (int32_t)((uint32_t)e.x & ~kStageMirror);
                const unsigned bm = __ballot_sync(0xffffffffu, m);
                const unsigned long long p1 = base + (unsigned long long)i;
                const unsigned long long p2 = mb + (unsigned long long)__popc(bm & lt);
                const int32_t pa = __shfl_sync(0xffffffffu, mine, i < ne ? (int)((p1 >> B.page_log2) - pg0) : 0);
                const int32_t pb = __shfl_sync(0xffffffffu, mine, m ? (int)((p2 >> B.page_log2) - pg0) : 0);
                if (i < ne && pa >= 0)
                    B.pool[((long long)pa << B.page_log2) | (long long)(p1 & mask)] = make_int2(qi, e.y);
                if (m && pb >= 0) B.pool[((long long)pb << B.page_log2) | (long long)(p2 & mask)] = make_int2(e.y, qi);
                mb += (unsigned long long)__popc(bm);
            }
        }
    } else {
        if (lane == 0 && total > 0) base = atomicAdd(&P.counters[1], total);
        base = __shfl_sync(0xffffffffu, base, 0);
        unsigned long long mb = base + (unsigned long long)ne;
        for (int i0 = 0; i0 < ne; i0 += 32) {
            const int i = i0 + lane;
            const int2 e = i < ne ? st.pairs[i] : make_int2(0, 0);
            const bool m = i < ne && ((uint32_t)e.x & kStageMirror) != 0u;
            const int32_t qi = (int32_t)((uint32_t)e.x & ~kStageMirror);
            const unsigned bm = __ballot_sync(0xffffffffu, m);
            const unsigned long long p1 = base + (unsigned long long)i;
            if (i < ne && p1 < P.capacity) P.out_pairs[p1] = make_int2(qi, e.y);
            const unsigned long long p2 = mb + (unsigned long long)__popc(bm & lt);
            if (m && p2 < P.capacity) P.out_pairs[p2] = make_int2(e.y, qi);
            mb += (unsigned long long)__popc(bm);
        }
    }
    __syncwarp();
    st.cnt = 0;
    if (lane == 0) W.smir = 0;
}

// Warp-collective: each lane offers nout in {0, 1, 2} pairs ((qid, cid) and,
// when 2, the mirrored (cid, qid)): one stage entry each, flagged when 2.
template <bool BATCH = true, typename W_t>
__device__ __forceinline__ void f32s_emit(W_t& W, WarpStage& st, const JoinParams& P, int lane,
                                          int nout, int32_t qid, int32_t cid) {
    const unsigned lt = (1u << lane) - 1u;
    const unsigned b1 = __ballot_sync(0xffffffffu, nout >= 1);
    const unsigned b2 = __ballot_sync(0xffffffffu, nout == 2);
    const int ne = __popc(b1);
    if (ne == 0) return;
    if (st.cnt + ne > st.cap) f32s_flush<BATCH>(W, st, P, lane);
    if (nout >= 1)
        st.pairs[st.cnt + __popc(b1 & lt)] =
            make_int2((int32_t)((uint32_t)qid | (nout == 2 ? kStageMirror : 0u)), cid);
    st.cnt += ne;
    if (lane == 0) W.smir += __popc(b2);
}

}  // namespace sj
