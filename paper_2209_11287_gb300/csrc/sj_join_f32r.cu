// The certified FP32 filter for small dimensions (padded d <= 8, without
// distances) on sparse indexes: cells of one or two points, as when
// near-duplicates of a large set are sought.
//
// Per pair it computes what k_join_f32s does (the same value, thresholds,
// recheck queue and stage).  That kernel gives a warp one work item at a time:
// it loads up to 16 queries, takes their bounding box, prefixes the item's runs
// and then evaluates chunks of 64 candidates.  With 1.4 queries and 31
// candidates an item those preparations are nearly all of the work (about 800
// instructions an item), and the box prunes no more than the evaluation itself.
// Here a warp takes kF32rItems items together: the runs of all of them are
// prefixed once, and the lanes take consecutive candidates of that list,
// whichever item they belong to; a lane finds its run among the at most 32
// that follow the chunk's first one and walks its own item's queries.  Bound by
// instruction issue.  Measured (1,000,001 uniform 4-D points, 4 neighbours,
// 692,967 items): 687 / 274 us.
#include <algorithm>
#include <atomic>

#include "sj_f32_stage.cuh"

namespace sj {

namespace {

constexpr int kF32rItems = 8;     // most items a warp takes at a time
constexpr int kF32rQ = 3;         // most queries of an item dealt with here when there is a list for the others
constexpr int kF32rRuns = 256;    // runs of a group of them (an item has at most kMaxRuns)
constexpr int kF32rStage = 256;
constexpr int kF32rWarps = 4;
static_assert(kMaxRuns <= kF32rRuns, "a group holds at least one item");
static_assert(2 * kF32rStage <= kStageMax, "a stage flush (entries and mirrors) resolves at most 32 pages");

struct F32rWarp {
    int32_t rstart[kF32rRuns];     // per run of the group: first sorted position,
    uint32_t rpre[kF32rRuns + 1];  // prefix of the lengths,
    uint8_t rmeta[kF32rRuns];      // item of the group | flag << 4 (0 plain, 1 mirrored, 2 self-cell triangle)
    int2 iq[kF32rItems];           // per item: its queries [x, y)
    int32_t ipre[kF32rItems + 1];  // prefix of the items' runs in the group
    int32_t ir0[kF32rItems];       // first run
    unsigned long long rechecked;  // pairs re-decided in place, queue full (lane 0)
    int smir;                      // staged entries flagged for a mirrored copy (lane 0)
    int2 stage[kF32rStage];
};

// TAKE: items a warp takes at a time (8, fewer where all warps would not get as
// many; a run-time number spilled for padded d = 8: 1,000,000 x 5-D 811 / 851 us).
template <int DP, int TAKE>
__global__ void __launch_bounds__(32 * kF32rWarps) k_join_f32r(JoinParams P) {
    __shared__ F32rWarp smem[kF32rWarps];
    const float* __restrict__ Y = static_cast<const float*>(P.y);
    const float* __restrict__ H = static_cast<const float*>(P.h);
    const int lane = threadIdx.x & 31;
    F32rWarp& W = smem[threadIdx.x >> 5];
    WarpStage st{W.stage, nullptr, 0, 0, kF32rStage};
    if (lane == 0) {
        W.rechecked = 0;
        W.smir = 0;
    }
    for (;;) {
        long long first = 0;
        if (lane == 0) first = (long long)atomicAdd(&P.counters[0], (unsigned long long)TAKE);
        first = __shfl_sync(0xffffffffu, first, 0);
        if (first >= P.n_items) break;
        const int have = (int)min((long long)TAKE, P.n_items - first);
        Item I{0, 0, 0, 0};
        if (lane < have) I = P.items[first + lane];
        if (!SJ_BOUND(P, I.q0 >= 0 && I.q1 <= P.n_points && I.r1 - I.r0 <= kF32rRuns, 51)) I = Item{0, 0, 0, 0};
        if (P.big_items) {  // items of many queries are left to k_join_f32s
            const bool big = I.q1 - I.q0 > kF32rQ;
            const unsigned m = __ballot_sync(0xffffffffu, big);
            if (m) {
                unsigned long long at = 0;
                if (lane == 0) at = atomicAdd(&P.counters[9], (unsigned long long)__popc(m));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (big) {
                    P.big_items[at + __popc(m & ((1u << lane) - 1u))] = (int32_t)(first + lane);
                    I = Item{0, 0, 0, 0};
                }
            }
        }
        int upto = I.r1 - I.r0;  // inclusive prefix of the items' runs
#pragma unroll
        for (int o = 1; o < kF32rItems; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += u;
        }
        for (int j0 = 0, taken = 0; j0 < have;) {  // groups of items whose runs fit
            const unsigned fit = __ballot_sync(0xffffffffu, lane >= j0 && lane < have && upto - taken <= kF32rRuns);
            const int nj = __popc(fit);  // (consecutive from j0, at least one)
            __syncwarp();
            if (lane >= j0 && lane < j0 + nj) {
                W.iq[lane - j0] = make_int2(I.q0, I.q1);
                W.ir0[lane - j0] = I.r0;
                W.ipre[lane - j0 + 1] = upto - taken;
            }
            if (lane == 0) W.ipre[0] = 0;
            __syncwarp();
            const int nruns = W.ipre[nj];
            uint32_t carry = 0;
            for (int b = 0; b < nruns; b += 32) {
                const int f = b + lane;
                uint32_t len = 0;
                if (f < nruns) {
                    int j = 0;
                    while (W.ipre[j + 1] <= f) ++j;
                    const Run R = P.runs[W.ir0[j] + f - W.ipre[j]];
                    const bool self = P.tri && !(R.end_flags & kMirrorBit);
                    const int32_t start = self ? W.iq[j].x : R.start;
                    W.rstart[f] = start;
                    W.rmeta[f] = (uint8_t)(j | (self ? 2 : (int)(R.end_flags >> 31)) << 4);
                    len = (uint32_t)((int32_t)(R.end_flags & ~kMirrorBit) - start);
                }
                uint32_t v = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += u;
                }
                if (f < nruns) W.rpre[f + 1] = carry + v;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (lane == 0) W.rpre[0] = 0;
            __syncwarp();
            const uint32_t C = carry;
            int run0 = 0;  // the run of the chunk's first candidate
            for (uint32_t v0 = 0; v0 < C; v0 += 32) {
                const uint32_t v = v0 + (uint32_t)lane;
                if (W.rpre[run0 + 1] <= v0) ++run0;  // (the last chunk ended with its run)
                // the last run r with rpre[r] <= v (runs are not empty, so it is
                // one of the 32 from the first candidate's on)
                int lo = run0, hi = min(run0 + 31, nruns - 1);
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    const int mid = (lo + hi + 1) >> 1;
                    const bool up = W.rpre[mid] <= v;
                    lo = up ? mid : lo;
                    hi = up ? hi : mid - 1;
                }
                run0 = __shfl_sync(0xffffffffu, lo, 31);
                const bool valid = v < C;
                int32_t j = 0, q = 0, qe = 0, cid = 0;
                int fl = 0;
                float c[DP], to = INFINITY, ti = INFINITY;
                if (valid) {
                    const uint32_t meta = W.rmeta[lo];
                    const int2 iq = W.iq[meta & 15u];
                    fl = (int)(meta >> 4);
                    j = W.rstart[lo] + (int32_t)(v - W.rpre[lo]);
                    if (!SJ_BOUND(P, j >= 0 && j < P.n_points, 52)) j = 0;
                    q = iq.x;
                    qe = fl == 2 ? min(iq.y, j + 1) : iq.y;  // (the triangle: queries up to the candidate)
                    load_coords<DP>(Y, j, c);
                    const float4 ax = P.aux[j];
                    to = ax.x;
                    ti = ax.y;
                    cid = __float_as_int(ax.z);
                } else {
#pragma unroll
                    for (int k = 0; k < DP; ++k) c[k] = 0.f;
                }
                while (__any_sync(0xffffffffu, q < qe)) {
                    int nout = 0;
                    int32_t qid = 0;
                    bool band = false, mir = false;
                    if (q < qe) {
                        float y[DP];
                        load_coords<DP>(Y, q, y);
                        float a = H[q];
#pragma unroll
                        for (int k = 0; k < DP; ++k) a = __fmaf_rn(y[k], c[k], a);
                        if (a >= to) {
                            mir = fl != 0 && q != j;
                            if (a >= ti) {
                                nout = mir ? 2 : 1;
                                qid = P.perm[q];
                            } else {
                                band = true;
                            }
                        }
                    }
                    if (__any_sync(0xffffffffu, band)) {
                        const bool queued = band_push(P, lane, band, q, j, mir);
                        const bool here = band && !queued;
                        const unsigned inplace = __ballot_sync(0xffffffffu, here);
                        if (lane == 0 && inplace) W.rechecked += (unsigned long long)__popc(inplace);
                        if (here && direct_sq(P.xs + (int64_t)q * P.dp, P.xs + (int64_t)j * P.dp, P.d) <= P.e2) {
                            nout = mir ? 2 : 1;
                            qid = P.perm[q];
                        }
                    }
                    f32s_emit<false>(W, st, P, lane, nout, qid, cid);
                    ++q;
                }
            }
            j0 += nj;
            taken = __shfl_sync(0xffffffffu, upto, j0 - 1);
        }
    }
    f32s_flush<false>(W, st, P, lane);
    if (lane == 0 && W.rechecked) atomicAdd(&P.counters[2], W.rechecked);
}

template <int DP, int TAKE>
int launch_f32r_dt(Index* ix, const JoinParams& p, double items) {
    auto kern = k_join_f32r<DP, TAKE>;
    static std::atomic<int> cached{0};  // resident CTAs per SM (a property of the kernel)
    int per_sm = cached.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        SJ_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kF32rWarps, 0));
        if (per_sm < 1) per_sm = 1;
        cached.store(per_sm, std::memory_order_relaxed);
    }
    const double need = items / (TAKE * kF32rWarps) + 1.0, most = (double)device_sm_count(ix->device) * per_sm;
    kern<<<(unsigned)(need < most ? need : most), 32 * kF32rWarps, 0, ix->stream>>>(p);
    note_launch();
    SJ_CK(cudaGetLastError());
    return SJ_OK;
}

// Items a warp takes: as many as give every warp of the chip (8 CTAs an SM) some
// at once, but 8 of items with few evaluations, whose warps cost more than their
// items (atomics on the queue and the cursor).  (4-D 3,000 points, 31 evaluations
// an item: 8 at a time 20.9 us, 1 12.5; 2-D 10,000, 2 evaluations: 8 at a time
// 10.5 us, 2 14.8.)
template <int DP>
int launch_f32r_d(Index* ix, const JoinParams& p, double items, bool light) {
    const double warps = (double)device_sm_count(ix->device) * 8 * kF32rWarps;
    if (items > 4 * warps || (light && items >= 2048)) return launch_f32r_dt<DP, 8>(ix, p, items);
    if (items > 2 * warps) return launch_f32r_dt<DP, 4>(ix, p, items);
    if (items > warps) return launch_f32r_dt<DP, 2>(ix, p, items);
    return launch_f32r_dt<DP, 1>(ix, p, items);
}

}  // namespace

// Taken for single joins whose cells are sparse, by the queries q and the
// evaluations e of an item and the number of items, counted as cells + n / 16
// (the part of them that a range of items is).  The lines were fitted to 545
// states (uniform and clustered, 2-D to 8-D, 1 to 40 neighbours, 300 to 1,000,000
// points) so that none is slower than k_join_f32s by more than 4%; tile us,
// k_join_f32s / this kernel alone / shared.
// Evenly filled cells (a point's own cell holds at most 1.4 times the mean
// cell; 1.6 in the plane from 2^17 items on: clusters 1,000,000, ratio 1.57, 867 /
// 649 / 685), this kernel alone.  Padded d <= 4: q < 2.5, and e < 160 from 2^16 items
// on (uniform 4-D 1,000,000 points: q 1.3 677 / 267, q 1.7, e 102 551 / 349, q
// 2.3, e 207 460 / 423; 3-D 300,000, q 4.1 89 / 142), else e < 60 (4-D 3,000, e 31
// 14.8 / 12.5; 1,000, e 85 13.2 / 14.5).  Padded d = 8: q < 1.9, and e < 250 from
// 2^17 items on (5-D 1,000,000: e 99 1187 / 639; 6-D, q 1.8, e 732 1771 / 1947),
// else e < 60 (6-D 10,000: e 77 29 / 24, e 185 34 / 41).
// Other cells, the items of up to 3 queries, where there are enough of them for
// two launches: 2^17 items, q < 2.5, e < 600, for d = 8 400 (clusters over noise,
// 3-D 342,000 items 520 / 1120 / 472, 4-D 511,000 588 / 606 / 432, 134,000 183 / 330 / 180,
// 49,000 76 / 162 / 93, 3-D 811 17 / 25 / 28).  (Batched joins and the filter's
// recording mode keep k_join_f32s.)
static double f32r_items(const Index* ix, double share) { return ((double)ix->n_cells + (double)ix->n / kQMax) * share; }

SparseUse f32r_use(const Index* ix, const JoinParams& p, double share) {
    if (p.batch || p.dbg || ix->n_cells <= 0) return SparseUse::none;
    const double n = (double)ix->n, cells = (double)ix->n_cells, items = f32r_items(ix, share);
    const double q = n / f32r_items(ix, 1.0), e = (double)ix->n_evaluated / f32r_items(ix, 1.0);
    const bool large = items >= (1 << 17);
    if ((double)ix->sum_sq / n > (ix->dp == 2 && large ? 1.6 : 1.4) * n / cells)
        return large && q < 2.5 && e < (ix->dp <= 4 ? 600.0 : 400.0) ? SparseUse::few_queries : SparseUse::none;
    const bool take = ix->dp <= 4 ? q < 2.5 && e < (items >= (1 << 16) ? 160.0 : 60.0)
                                  : q < 1.9 && e < (large ? 250.0 : 60.0);
    return take ? SparseUse::all : SparseUse::none;
}

int launch_join_f32r(Index* ix, const JoinParams& p, double share) {
    const double items = f32r_items(ix, share);
    const bool light = (double)ix->n_evaluated < 8.0 * f32r_items(ix, 1.0);
    switch (ix->dp) {
        case 2: return launch_f32r_d<2>(ix, p, items, light);
        case 4: return launch_f32r_d<4>(ix, p, items, light);
        case 8: return launch_f32r_d<8>(ix, p, items, light);
        default:
            set_error("no small-d FP32 kernel for padded dimension %d", ix->dp);
            return SJ_ERR_UNSUPPORTED;
    }
}

}  // namespace sj
