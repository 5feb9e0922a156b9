// What the tensor-core filter leaves open: its records (one candidate against
// up to 32 query positions, see sj_join_tc.cu) become result pairs.
//
// The filter's tile kernel only finds the maybe-in pairs and appends a record
// where there are any; deciding and emitting them there kept each epilogue warp
// in long serial code while its accumulator waited (16-D mixture, 500,000
// points: 2.2 of 5.2 ms).  Here they are spread over the whole chip: a warp
// expands 32 records into a list and deals with 32 pairs at a time.
//
// A pair that the filter's bound does not certify is first evaluated in
// binary32 by the direct form on the kernel coordinates, sum of (y_q - y_c)^2.
// That sum's error is relative to the distance, not to the norms of the points
// as in the expanded form, so nearly every pair is certified out or in by it
// (refine_out, refine_in; pack_coefficients), at FP32 rate; binary64, which
// runs at 1/64 of that, decides the rest and gives the distances.  Measured
// against rechecking every such pair in binary64 (k_recheck, with the emission
// of the certain pairs still in the tile kernel): 500,000 x 16-D mixture (7.3 M
// uncertain of 28 M pairs) 703 / 380 us, 200,000 x 64-D 586 / 210 us.  Bound by
// the gathers of rows and ids and the emission.
#include "sj_join_common.cuh"

namespace sj {

namespace {

constexpr int kResolveWarps = 4;
constexpr int kResolveBlocks = 8;
constexpr int kResolveRun = 16;  // blocks of 32 records that one warp takes in a row, at most

// Squared distance of two kernel-coordinate rows, binary32.
template <int DP>
__device__ __forceinline__ float refine_sq(const float* __restrict__ a, const float* __restrict__ b) {
    float s = 0.f;
    if constexpr (DP < 4) {
#pragma unroll
        for (int k = 0; k < DP; ++k) {
            const float t = a[k] - b[k];
            s = __fmaf_rn(t, t, s);
        }
    } else {
#pragma unroll 4
        for (int k = 0; k < DP / 4; ++k) {
            const float4 u = reinterpret_cast<const float4*>(a)[k], v = reinterpret_cast<const float4*>(b)[k];
            const float t0 = u.x - v.x, t1 = u.y - v.y, t2 = u.z - v.z, t3 = u.w - v.w;
            s = __fmaf_rn(t0, t0, s);
            s = __fmaf_rn(t1, t1, s);
            s = __fmaf_rn(t2, t2, s);
            s = __fmaf_rn(t3, t3, s);
        }
    }
    return s;
}

// Pairs of several batched instances in a warp: a reservation for each instance,
// its lanes one after another.  (Out of line: rare, and the kernel's registers
// are few: 2M x 4-D 670 us with it inlined three times, 634 so.)
__device__ __noinline__ void resolve_emit_mixed(const JoinParams& P, int lane, int gid, int nout, int32_t qid, int32_t cid,
                                                double dist) {
    const BatchJoin& B = *P.batch;
    const unsigned same = __match_any_sync(0xffffffffu, nout > 0 ? gid : -1);
    const unsigned two = __ballot_sync(0xffffffffu, nout == 2), lt = (1u << lane) - 1u;
    const int first = __ffs(same) - 1;
    unsigned long long at = 0;
    if (nout > 0 && lane == first)
        at = atomicAdd(&B.cursor[gid], (unsigned long long)(__popc(same) + __popc(same & two)));
    at = __shfl_sync(0xffffffffu, at, first) + (unsigned)(__popc(same & lt) + __popc(same & two & lt));
    for (int u = 0; u < nout; ++u) {
        const long long slot = batch_slot(B, gid, at + (unsigned)u);
        if (slot < 0) continue;
        B.pool[slot] = u == 0 ? make_int2(qid, cid) : make_int2(cid, qid);
        if (P.emit_dist) B.dpool[slot] = dist;
    }
}

// Bound by the latency of its gathers (positions to ids and rows, cursor and
// page of a flush), so a pair's first loads do not wait for one another
// (500,000 x 16-D mixture, build, filter and this kernel: the ids loaded after
// the decision 2.69 ms, before it 2.64).  8 CTAs an SM leave 64 registers a
// thread; 10, 12 and 16 were slower (2.73, 2.81 ms and more, by the spills).
template <int DP, bool EMIT>
__global__ void __launch_bounds__(32 * kResolveWarps, kResolveBlocks) k_resolve(JoinParams P) {
    __shared__ int2 s_stage[kResolveWarps][kStage];
    __shared__ double s_sdist[kResolveWarps][EMIT ? kStage : 1];
    // pairs waiting: (query position | certain << 31, candidate position | mirrored << 31)
    __shared__ int2 s_list[kResolveWarps][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float* __restrict__ Y = static_cast<const float*>(P.y);
    WarpStage st{s_stage[wid], EMIT ? s_sdist[wid] : nullptr, 0, 0};
    int2* list = s_list[wid];
    int waiting = 0;
    unsigned long long decided = 0;
    const int32_t* __restrict__ inst_of = P.batch ? P.batch->inst_of_sorted : nullptr;
    const int32_t* __restrict__ inst_gid = P.batch ? P.batch->inst_gid : nullptr;
    const long long* __restrict__ inst_off = P.batch ? P.batch->inst_off : nullptr;

    // 32 pairs, one a lane
    auto deal = [&](bool live, int2 e) {
        const int32_t qs = (int32_t)((uint32_t)e.x & ~kMirrorBit), cs = (int32_t)((uint32_t)e.y & ~kMirrorBit);
        live = live && SJ_BOUND(P, qs < P.n_points && cs < P.n_points, 41);
        const bool certain = e.x < 0;
        int nout = 0, gid = 0;
        int32_t qid = 0, cid = 0;
        double dist = 0.0;
        if (live) {
            qid = P.perm[qs];
            cid = P.perm[cs];
            const int li = inst_of ? inst_of[qs] : 0;
            bool in = certain;
            if (EMIT || !certain) {
                ++decided;
                bool exact = EMIT;  // (the binary64 sum is needed)
                if (!certain) {
                    const float s32 = refine_sq<DP>(Y + (int64_t)qs * DP, Y + (int64_t)cs * DP);
                    const float2 r = inst_of ? P.batch->inst_refine[li] : make_float2(P.refine_out, P.refine_in);
                    in = s32 < r.y;
                    exact = (EMIT || !in) && !(s32 > r.x);
                }
                if (exact) {
                    const double s = direct_sq(P.xs + (int64_t)qs * DP, P.xs + (int64_t)cs * DP, P.d);
                    in = s <= (inst_of ? P.batch->inst_e2[li] : P.e2);
                    if (EMIT && in) dist = sqrt(s);
                }
            }
            if (in) nout = e.y < 0 && cs != qs ? 2 : 1;
            if (inst_of) {
                gid = inst_gid[li];
                const int32_t off = (int32_t)inst_off[li];
                qid -= off;
                cid -= off;
            }
        }
        if (P.batch) {
            // the pairs of a warp that belong to one instance share its stage;
            // those of several are written here, with a reservation for each
            // instance (one for each pair: 409 us for the 2.4 M pairs of 64
            // planar joins of 2,000 points, all on 64 cursors; 61 us so)
            const unsigned some = __ballot_sync(0xffffffffu, nout > 0);
            if (some == 0u) return;
            const int g0 = __shfl_sync(0xffffffffu, gid, __ffs(some) - 1);
            if (!__all_sync(0xffffffffu, nout == 0 || gid == g0)) {
                resolve_emit_mixed(P, lane, gid, nout, qid, cid, dist);
                __syncwarp();
                return;
            }
            if (st.cnt > 0 && st.gid != g0) stage_flush(st, P, lane);
            st.gid = g0;
        }
        if (EMIT)
            stage_emit(st, P, lane, nout, qid, cid, dist);
        else
            stage_emit_pairs(st, P, lane, nout, qid, cid);
    };

    const int4* __restrict__ records = reinterpret_cast<const int4*>(P.band);
    const unsigned long long taken = P.counters[3], room = P.band_cap >> 1;
    const unsigned long long count = taken < room ? taken : room;
    // A warp takes up to kResolveRun blocks of 32 records that follow one
    // another: in a batch they come from the same few instances, so the stage
    // fills before the instance changes (blocks a grid apart changed it nearly
    // every time: a flush, with its atomic on the instance's cursor, for 32
    // records, and a warp of mixed leftovers written pair by pair).  Measured,
    // 96 joins in one batch: blocks a grid apart 6.52 ms, runs of 4 6.22, 16
    // 6.19, 64 6.17; one join of the 16-D mixture 2.64 / 2.67 / 2.67 / 2.77 ms,
    // long runs leave warps idle.
    // With distances few records are spread over all warps in blocks of fewer (a
    // block's pairs are dealt with 32 at a time, one after another, and each takes
    // the latency of its binary64 sums).  4,000 x 64-D points with
    // distances, 61,000 pairs, filter and this kernel: 188 us with blocks of 32
    // and every pair in binary32 first, 128 so and with the certain ones in
    // binary64 at once.
    const unsigned long long warps = (unsigned long long)gridDim.x * kResolveWarps;
    int size = 32;  // records of a block
    if constexpr (EMIT)
        while (size > 8 && count < warps * (unsigned)(size / 2)) size >>= 1;
    const unsigned long long blocks = (count + (unsigned)size - 1) / (unsigned)size;
    const unsigned long long run = min((unsigned long long)kResolveRun, max(1ull, blocks / (2 * warps)));
    int of_list = -1;  // batch: the instance of the waiting pairs
    unsigned long long r = (unsigned long long)blockIdx.x * kResolveWarps + wid, k_run = 0;
    for (; r * run + k_run < blocks; k_run + 1 < run ? ++k_run : (k_run = 0, r += warps)) {
        const unsigned long long b = (r * run + k_run) * (unsigned)size;
        const int4 e = (!EMIT || lane < size) && b + lane < count ? records[b + lane] : make_int4(0, 0, 0, 0);
        if (inst_of) {  // what waits of another instance goes first, so that a warp of pairs has one
            const int cs = (int)((uint32_t)e.w & ~kMirrorBit);
            const unsigned some = __ballot_sync(0xffffffffu, e.x != 0);
            if (some == 0u) continue;
            int li = e.x != 0 && SJ_BOUND(P, cs < P.n_points, 41) ? inst_of[cs] : 0;
            li = __shfl_sync(0xffffffffu, li, __ffs(some) - 1);
            if (waiting > 0 && li != of_list) {
                __syncwarp();
                deal(lane < waiting, list[lane < waiting ? lane : 0]);
                __syncwarp();
                waiting = 0;
            }
            of_list = li;
        }
        uint32_t m = (uint32_t)e.x;
        for (;;) {  // a column of every record at a time into the list
            const unsigned w = __ballot_sync(0xffffffffu, m != 0u);
            if (w == 0u) break;
            if (m) {
                const int k = __ffs(m) - 1;
                m &= m - 1u;
                list[waiting + __popc(w & ((1u << lane) - 1u))] =
                    make_int2((int)((uint32_t)(e.z + k) | ((uint32_t)e.y >> k & 1u) << 31), e.w);
            }
            waiting += __popc(w);
            if (waiting >= 32) {
                waiting -= 32;
                __syncwarp();
                deal(true, list[waiting + lane]);
                __syncwarp();
            }
        }
    }
    __syncwarp();
    deal(lane < waiting, list[lane < waiting ? lane : 0]);
    stage_flush(st, P, lane);
    for (int o = 16; o > 0; o >>= 1) decided += __shfl_down_sync(0xffffffffu, decided, o);
    if (lane == 0 && decided) atomicAdd(&P.counters[2], decided);
}

template <int DP>
int launch_resolve_dp(Index* ix, const JoinParams& p) {
    const unsigned blocks = (unsigned)device_sm_count(ix->device) * kResolveBlocks;
    if (p.emit_dist)
        k_resolve<DP, true><<<blocks, 32 * kResolveWarps, 0, ix->stream>>>(p);
    else
        k_resolve<DP, false><<<blocks, 32 * kResolveWarps, 0, ix->stream>>>(p);
    note_launch();
    SJ_CK(cudaGetLastError());
    return SJ_OK;
}

}  // namespace

int launch_resolve(Index* ix, const JoinOut& out, int emit_dist) {
    const JoinParams p = make_join_params(ix, out, emit_dist);
    switch (ix->dp) {
        case 2: return launch_resolve_dp<2>(ix, p);
        case 4: return launch_resolve_dp<4>(ix, p);
        case 8: return launch_resolve_dp<8>(ix, p);
        case 16: return launch_resolve_dp<16>(ix, p);
        case 32: return launch_resolve_dp<32>(ix, p);
        case 64: return launch_resolve_dp<64>(ix, p);
        default:
            set_error("no record resolution for padded dimension %d", ix->dp);
            return SJ_ERR_UNSUPPORTED;
    }
}

}  // namespace sj
