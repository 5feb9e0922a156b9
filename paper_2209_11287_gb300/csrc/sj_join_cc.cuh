// Distance tiles on CUDA cores, fused with the eps threshold and the
// compaction into result pages (templates; each padded dimension is
// instantiated in a translation unit of its own, sj_cc_d*.cu, so the library
// compiles in parallel).
//
// One work item = up to kQMax queries of one grid cell and the candidate runs
// of that cell (Sec. III-B: the queries of a cell share their candidates).
// Per (query, candidate) pair the tile computes, in the kernel type T,
//     a = -||y_q||^2 / 2 + sum_k y_qk * y_ck          (fma chain, k ascending)
// which is the expanded form of Eq. 3 with the constant part moved to the
// candidate's threshold: ||y_q - y_c||^2 = ||y_c||^2 - 2 a.  Per-candidate
// thresholds (computed at packing) certify the decision: a < thr_out means
// out, a >= thr_in means in; pairs in between are re-decided with the
// decision rule itself (binary64 direct form, dimension order, no
// contraction) by k_recheck, so the returned set equals the rule's.
//
// T = double is the plain FP64 join (Eq. 3/4 evaluated on FP64 CUDA cores);
// T = float is the certified FP32 filter.
//
// Work decomposition: every warp takes work items on its own (an atomic
// queue, the next index fetched one item ahead), so no block-wide barrier
// ever stalls a tile.  A warp evaluates its item in chunks of 32 x TC
// candidates: each lane holds TC candidates in registers and walks the
// item's queries, broadcast from shared memory.  For d <= 8 the threshold
// test is fused into the query loop (and FP32 pairs of candidates use the
// paired FMA, one rounding per lane as for the scalar FMA); for larger d
// the accumulators of all queries are kept and tested after the d-loop.  The
// "maybe in" pairs of a chunk (a >= thr_out) are compacted into a per-warp
// list with one warp scan, and the list is classified 32 entries at a time,
// so the rare work (certain-in test, queueing for the recheck, emission)
// runs with every lane busy.
#pragma once

#include <type_traits>

#include "sj_join_common.cuh"

namespace sj {

// Warps per CTA (independent of each other): as many as keep the per-warp
// shared memory of a CTA within the 48 KB of static shared memory, at most 4.
template <typename WS>
constexpr int cc_warps() {
    return sizeof(WS) * 4 <= 46 * 1024 ? 4 : sizeof(WS) * 2 <= 46 * 1024 ? 2 : 1;
}

template <typename T, int DP, int TC, bool EMIT, int RUNS, bool PRUNE>
struct CcWarpSmem {
    ItemSmem<T, DP, RUNS> it;
    int32_t cj[EMIT ? 32 * TC : 1];    // sorted position of each candidate slot (with distances)
    int32_t cperm[32 * TC];            // its input index
    uint8_t cmir[32 * TC];             // its mirror flag
    uint16_t list[EMIT ? 32 * TC * (kQMax / 2) : 1];  // with distances: maybe-in entries of one half
                                                      // of the queries, slot << 4 | query
    int2 stage[kStage];
    double sdist[EMIT ? kStage : 1];
    double scq[DP >= 16 ? kQMax : 1];  // short-circuit: each query's w
    // candidates kept by the bounding-box prune (position, run flag), and the
    // box of the item's queries
    static constexpr uint32_t RING = 32 * TC - 1 + 64 <= 128 ? 128 : 256;
    int32_t ring_j[PRUNE ? RING : 1];
    uint8_t ring_f[PRUNE ? RING : 1];
    float blo[PRUNE ? DP : 1], bhi[PRUNE ? DP : 1];
    unsigned long long pruned;  // evaluations that the prune removed (lane 0; not in a register: FP64 has none to spare)
};

// Compaction step of the prune, d <= 8: candidates [v0, v0 + 64) of the item,
// two a lane, against the box of its queries; the kept ones follow the ring's
// `cnt` entries from `head`.  The same lossless test as k_join_f32s
// (f32s_gather: a lower bound of the squared distance to the box, every
// operation rounded down, against the radius behind the certified "out"
// threshold), here in front of the tiles with distances and the FP64 tile where
// cc_prune says so.
// The latter's binary64 coordinates are rounded to binary32 for it, which its
// radius allows for (fp64_prune_r2).  `r` is the lane's run cursor.
// A radius of +inf keeps everything.  Returns the candidates dropped.  Measured,
// FP64 tile with distances (200,000 uniform 4-D points, 64 neighbours, 9 queries
// an item; FP64 pipe): 705 us over all candidates, 495 us behind the prune.
template <typename T, int DP, int TC, bool EMIT, int RUNS>
__device__ __forceinline__ uint32_t cc_gather(CcWarpSmem<T, DP, TC, EMIT, RUNS, true>& W, const JoinParams& P, float r2,
                                              uint32_t C, uint32_t v0, int lane, int& r, uint32_t head, uint32_t& cnt) {
    constexpr uint32_t RING = CcWarpSmem<T, DP, TC, EMIT, RUNS, true>::RING;
    const T* __restrict__ Y = static_cast<const T*>(P.y);
    ItemSmem<T, DP, RUNS>& S = W.it;
    int32_t jj[2];
    uint32_t f[2];
    bool keep[2], test[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const uint32_t v = v0 + (uint32_t)(32 * g + lane);
        jj[g] = 0;
        f[g] = 0;
        keep[g] = v < C;
        if (v < C) {
            while (S.rpre[r + 1] <= v) ++r;
            jj[g] = S.rstart[r] + (int32_t)(v - S.rpre[r]);
            if (!SJ_BOUND(P, jj[g] >= 0 && jj[g] < P.n_points && r < RUNS, 21)) jj[g] = 0;
            f[g] = S.rmir[r];
        }
        test[g] = keep[g] && f[g] != 2u && r2 < INFINITY;
    }
    float c[2][DP];
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
        for (int k = 0; k < DP; ++k) c[g][k] = test[g] ? (float)Y[(int64_t)jj[g] * DP + k] : 0.f;
    uint32_t kept = 0;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        float lb = 0.f;
#pragma unroll
        for (int k = 0; k < DP; ++k) {
            const float gap = fmaxf(fmaxf(__fsub_rd(W.blo[k], c[g][k]), __fsub_rd(c[g][k], W.bhi[k])), 0.f);
            lb = __fmaf_rd(gap, gap, lb);
        }
        if (test[g] && lb > r2) keep[g] = false;
        const unsigned m = __ballot_sync(0xffffffffu, keep[g]);
        if (keep[g]) {
            const uint32_t e = (head + cnt + kept + (uint32_t)__popc(m & ((1u << lane) - 1u))) & (RING - 1u);
            W.ring_j[e] = jj[g];
            W.ring_f[e] = (uint8_t)f[g];
        }
        kept += (uint32_t)__popc(m);
    }
    cnt += kept;
    return min(64u, C - v0) - kept;
}

// Maybe-in bitmasks of TC candidates against all queries of the item, d <= 8:
// the threshold test follows each query's fma chain.
template <typename T, int DP, int TC, int RUNS>
__device__ __forceinline__ void tile_fused(const ItemSmem<T, DP, RUNS>& S, int Q, const T (&c)[TC][DP], const T (&to)[TC],
                                           const T (&ti)[TC], uint32_t (&bits)[TC], uint32_t (&cbits)[TC]) {
#pragma unroll
    for (int t = 0; t < TC; ++t) bits[t] = cbits[t] = 0;
    if constexpr (std::is_same<T, float>::value && TC % 2 == 0) {
#pragma unroll
        for (int q = 0; q < kQMax; ++q) {
            if (q >= Q) break;
            const float h = S.qh[q];
#pragma unroll
            for (int t = 0; t < TC; t += 2) {
                float2 a = make_float2(h, h);
#pragma unroll
                for (int k = 0; k < DP; ++k) {
                    const float qv = S.qy[q][k];
                    a = __ffma2_rn(make_float2(qv, qv), make_float2(c[t][k], c[t + 1][k]), a);
                }
                if (a.x >= to[t]) bits[t] |= 1u << q;
                if (a.y >= to[t + 1]) bits[t + 1] |= 1u << q;
                if (a.x >= ti[t]) cbits[t] |= 1u << q;
                if (a.y >= ti[t + 1]) cbits[t + 1] |= 1u << q;
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < kQMax; ++q) {
            if (q >= Q) break;
            const T h = S.qh[q];
#pragma unroll
            for (int t = 0; t < TC; ++t) {
                T a = h;
#pragma unroll
                for (int k = 0; k < DP; ++k) a = fma_t(S.qy[q][k], c[t][k], a);
                if (ge_threshold(a, to[t])) bits[t] |= 1u << q;
                if (ge_threshold(a, ti[t])) cbits[t] |= 1u << q;
            }
        }
    }
}

// Emission of one chunk without distances.  Certain pairs (maybe-in and
// certain-in bits) go straight into the warp's stage: one warp scan of each
// lane's output count (two outputs for a mirrored pair, one for a self pair)
// gives every lane its slots, and each lane writes its pairs in query order.
// A chunk larger than the stage is written in stage-sized windows, each
// flushed when full.  Uncertain pairs (maybe-in, not certain-in: the
// certified bound straddles eps) are queued for the binary64 recheck, one
// per lane per round, or re-decided here when the queue is full.
template <int TC>
__device__ __forceinline__ void emit_direct(WarpStage& st, const JoinParams& P, const int32_t* cperm,
                                            const uint8_t* cmir, const int32_t* qids, const ItemRoute& R,
                                            const Item& I, int lane, const int32_t (&j)[TC],
                                            const uint32_t (&bits)[TC], const uint32_t (&cbits)[TC],
                                            unsigned long long& rechecked) {
    int nout = 0;
    uint32_t any_unc = 0;
#pragma unroll
    for (int t = 0; t < TC; ++t) {
        const uint32_t cin = bits[t] & cbits[t];
        any_unc |= bits[t] & ~cbits[t];
        if (cin) {
            const int fl = cmir[t * 32 + lane];
            const int c = __popc(cin);
            nout += fl ? 2 * c : c;
            const int qd = j[t] - I.q0;  // the diagonal of a self-cell candidate
            if (fl == 2 && qd >= 0 && qd < kQMax && ((cin >> qd) & 1u)) nout -= 1;
        }
    }
    int total;
    const int off = warp_excl_scan(nout, lane, &total);
    if (total > 0) {
        if (st.cnt + total > kStage) stage_flush(st, P, lane);
        for (int w0 = 0; w0 < total;) {  // warp-uniform
            const int w1 = min(total, w0 + (kStage - st.cnt));
            if (off < w1 && off + nout > w0) {
                int idx = off;
#pragma unroll
                for (int t = 0; t < TC; ++t) {
                    uint32_t b = bits[t] & cbits[t];
                    if (!b) continue;
                    const int slot = t * 32 + lane;
                    const int fl = cmir[slot];
                    const int32_t cid = (int32_t)(cperm[slot] - R.off);
                    const int qd = fl == 2 ? j[t] - I.q0 : -1;
                    while (b) {
                        const int q = __ffs(b) - 1;
                        b &= b - 1u;
                        const int32_t qid = (int32_t)(qids[q] - R.off);
                        if (idx >= w0 && idx < w1) st.pairs[st.cnt + idx - w0] = make_int2(qid, cid);
                        ++idx;
                        if (fl == 1 || (fl == 2 && q != qd)) {
                            if (idx >= w0 && idx < w1) st.pairs[st.cnt + idx - w0] = make_int2(cid, qid);
                            ++idx;
                        }
                    }
                }
            }
            st.cnt += w1 - w0;
            w0 = w1;
            if (st.cnt == kStage) stage_flush(st, P, lane);
        }
    }
    if (!__any_sync(0xffffffffu, any_unc != 0u)) return;
    uint32_t unc[TC];
#pragma unroll
    for (int t = 0; t < TC; ++t) unc[t] = bits[t] & ~cbits[t];
    for (;;) {
        bool want = false;
        int q = 0, slot = 0;
        int32_t jj = 0;
#pragma unroll
        for (int t = 0; t < TC; ++t)
            if (!want && unc[t]) {
                q = __ffs(unc[t]) - 1;
                unc[t] &= unc[t] - 1u;
                want = true;
                jj = j[t];
                slot = t * 32 + lane;
            }
        if (!__any_sync(0xffffffffu, want)) break;
        const int fl = want ? cmir[slot] : 0;
        const bool mir = fl == 1 || (fl == 2 && jj != I.q0 + q);
        const bool queued = band_push(P, lane, want, I.q0 + q, jj, mir);  // rare: no reservation
        int no = 0;
        int32_t qid = 0, cid = 0;
        if (want && !queued) {  // queue full: decide here
            const double s = direct_sq(P.xs + (int64_t)(I.q0 + q) * P.dp, P.xs + (int64_t)jj * P.dp, P.d);
            ++rechecked;
            if (s <= R.e2) {
                no = mir ? 2 : 1;
                qid = (int32_t)(qids[q] - R.off);
                cid = (int32_t)(cperm[slot] - R.off);
            }
        }
        stage_emit_pairs(st, P, lane, no, qid, cid);
    }
}

// Minimum resident CTAs per SM requested from the register allocator, and
// candidates per lane, of the FP32 small-d tile with distances (d <= 8): it is
// latency-bound, so it runs with 2 candidates per lane and 9 CTAs of 4 warps per
// SM (at most 56 registers); behind the bounding-box prune, which takes more
// registers, with 7 (200,003 uniform 3-D points, 48 neighbours: 9 CTAs, with
// spills, 156 us, 8 152, 7 150; without the prune 155).  Compile-time tuning
// constants.
#ifndef SJ_CC_F32_MIN_BLOCKS
#define SJ_CC_F32_MIN_BLOCKS 9
#endif
#ifndef SJ_CC_F32_PRUNE_MIN_BLOCKS
#define SJ_CC_F32_PRUNE_MIN_BLOCKS 7
#endif
#ifndef SJ_CC_TC_SMALL_D
#define SJ_CC_TC_SMALL_D 2
#endif
template <typename T, int DP, bool PRUNE>
constexpr int cc_min_blocks() {
    return !std::is_same<T, float>::value || DP > 8 ? 1 : PRUNE ? SJ_CC_F32_PRUNE_MIN_BLOCKS : SJ_CC_F32_MIN_BLOCKS;
}

// PRUNE (d <= 8): the candidates pass the bounding-box prune first (cc_prune).
template <typename T, int DP, int TC, bool EMIT, int NW, int RUNS, bool PRUNE>
__global__ void __launch_bounds__(NW * 32, cc_min_blocks<T, DP, PRUNE>()) k_join_cc(JoinParams P) {
    constexpr bool FUSED = DP <= 8;
    static_assert(FUSED || !PRUNE, "the prune is for small dimensions");
    constexpr int KC = DP < 8 ? DP : 8;  // dims per register chunk (unfused path)
    constexpr int SLOTS = 32 * TC;
    static_assert(SLOTS <= 2048, "slot index must fit in 11 bits");
    __shared__ CcWarpSmem<T, DP, TC, EMIT, RUNS, PRUNE> smem[NW];

    const T* __restrict__ Y = static_cast<const T*>(P.y);
    const T* __restrict__ TO = static_cast<const T*>(P.thr_out);
    const T* __restrict__ TI = static_cast<const T*>(P.thr_in);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    CcWarpSmem<T, DP, TC, EMIT, RUNS, PRUNE>& W = smem[wid];
    ItemSmem<T, DP, RUNS>& S = W.it;
    WarpStage st{W.stage, EMIT ? W.sdist : nullptr, 0, 0};
    BandQ bq{0, 0};
    unsigned long long rechecked = 0;
    if (PRUNE && lane == 0) W.pruned = 0;

    long long next = 0;
    if (lane == 0) next = (long long)atomicAdd(&P.counters[0], 1ull);
    next = __shfl_sync(0xffffffffu, next, 0);
    for (;;) {
        const long long it = next;
        if (it >= P.n_items) break;
        if (lane == 0) next = (long long)atomicAdd(&P.counters[0], 1ull);  // used next iteration
        next = __shfl_sync(0xffffffffu, next, 0);
        const Item I = P.items[it];
        const int Q = I.q1 - I.q0;
        const int nr = I.r1 - I.r0;
        const ItemRoute R = item_route(st, P, it, lane);
        const uint32_t C = load_item_warp<T, DP>(S, P, I, lane);
        if constexpr (std::is_same<T, double>::value && DP >= 16) {
            if (P.sc_w) {  // each query's remainder bound
                if (lane < kQMax) W.scq[lane] = lane < Q ? P.sc_w[I.q0 + lane] : 0.0;
                __syncwarp();
            }
        }

        if constexpr (PRUNE) {  // the box of the queries (32 is a multiple of DP: a lane keeps to one dim)
            float bmin = INFINITY, bmax = -INFINITY;
            for (int i = lane; i < Q * DP; i += 32) {
                const float v = (float)S.qy[i / DP][i % DP];
                bmin = fminf(bmin, v);
                bmax = fmaxf(bmax, v);
            }
#pragma unroll
            for (int o = DP; o < 32; o <<= 1) {
                bmin = fminf(bmin, __shfl_xor_sync(0xffffffffu, bmin, o));
                bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
            }
            if (lane < DP) {
                W.blo[lane] = bmin;
                W.bhi[lane] = bmax;
            }
            __syncwarp();
        }
        int run = 0;
        uint32_t head = 0, cnt = 0, v0 = 0;  // the ring; candidates gathered
        for (uint32_t base = 0;;) {
            uint32_t ns;  // candidates of this chunk
            if constexpr (PRUNE) {
                while (v0 < C && cnt < (uint32_t)SLOTS) {
                    const uint32_t out = cc_gather<T, DP, TC, EMIT, RUNS>(W, P, R.r2, C, v0, lane, run, head, cnt);
                    if (lane == 0) W.pruned += (unsigned long long)(out * (uint32_t)Q);
                    v0 += 64u;
                }
                if (cnt == 0) break;
                ns = min(cnt, (uint32_t)SLOTS);
                __syncwarp();
            } else {
                if (base >= C) break;
                ns = min(C - base, (uint32_t)SLOTS);
            }
            int32_t j[TC];
            bool valid[TC];
            uint32_t tri_mask[TC];
            T to[TC], ti[TC];
#pragma unroll
            for (int t = 0; t < TC; ++t) {
                const int slot = t * 32 + lane;
                valid[t] = (uint32_t)slot < ns;
                j[t] = 0;
                tri_mask[t] = 0xFFFFFFFFu;
                to[t] = T(INFINITY);  // an empty slot is never maybe-in
                ti[t] = T(INFINITY);
                if (valid[t]) {
                    uint8_t fl;
                    if constexpr (PRUNE) {
                        const uint32_t e = (head + (uint32_t)slot) & (CcWarpSmem<T, DP, TC, EMIT, RUNS, true>::RING - 1u);
                        j[t] = W.ring_j[e];
                        fl = W.ring_f[e];
                    } else {
                        j[t] = map_candidate_flag<T, DP>(S, nr, base + (uint32_t)slot, fl);
                        if (!SJ_BOUND(P, j[t] >= 0 && j[t] < P.n_points, 21)) j[t] = 0;
                    }
                    to[t] = TO[j[t]];
                    ti[t] = TI[j[t]];
                    if constexpr (EMIT) W.cj[slot] = j[t];
                    W.cperm[slot] = P.perm[j[t]];
                    W.cmir[slot] = fl;
                    // self-cell triangle: candidate j pairs with queries q0 .. j only
                    tri_mask[t] = (fl == 2 && j[t] < I.q1) ? (2u << (j[t] - I.q0)) - 1u : 0xFFFFFFFFu;
                }
            }
            uint32_t bits[TC], cbits[TC];
            if constexpr (FUSED) {
                T c[TC][DP];
#pragma unroll
                for (int t = 0; t < TC; ++t)
#pragma unroll
                    for (int k = 0; k < DP; ++k) c[t][k] = valid[t] ? Y[(int64_t)j[t] * DP + k] : T(0);
                tile_fused<T, DP, TC, RUNS>(S, Q, c, to, ti, bits, cbits);
            } else {
                T acc[TC][kQMax];
#pragma unroll
                for (int q = 0; q < kQMax; ++q)
#pragma unroll
                    for (int t = 0; t < TC; ++t) acc[t][q] = S.qh[q];
                bool all_out = false;  // short-circuit taken: every pair of the tile is out
#pragma unroll
                for (int kc = 0; kc < DP; kc += KC) {
                    T c[TC][KC];
#pragma unroll
                    for (int t = 0; t < TC; ++t)
#pragma unroll
                        for (int kk = 0; kk < KC; ++kk) c[t][kk] = valid[t] ? Y[(int64_t)j[t] * DP + kc + kk] : T(0);
#pragma unroll
                    for (int q = 0; q < kQMax; ++q) {
                        if (q >= Q) break;
#pragma unroll
                        for (int kk = 0; kk < KC; ++kk) {
                            const T qv = S.qy[q][kc + kk];
#pragma unroll
                            for (int t = 0; t < TC; ++t) acc[t][q] = fma_t(qv, c[t][kk], acc[t][q]);
                        }
                    }
                    if constexpr (std::is_same<T, double>::value && DP >= 16) {
                        // short-circuit (Sec. III-B) at the checkpoint, after the
                        // first sc_b dims: with w bounding half the remaining norm
                        // of each point (plus the rounding margins),
                        // acc + w_q + w_c below thr_out means the full filter value
                        // is below it too, i.e. the pair is certainly out; when that
                        // holds for every pair of the warp's tile the remaining
                        // dims are skipped
                        // (a one-pair-per-lane pre-test first: the full test runs
                        // only when that already holds for the whole warp)
                        if (P.sc_w && kc + KC == P.sc_b &&
                            __all_sync(0xffffffffu,
                                       !valid[0] || order_key(__dadd_ru(acc[0][0], W.scq[0])) <
                                                        order_key(__dsub_rd(to[0], P.sc_w[j[0]])))) {
                            bool out = true;
#pragma unroll
                            for (int t = 0; t < TC; ++t) {
                                if (!valid[t]) continue;
                                const long long kr = order_key(__dsub_rd(to[t], P.sc_w[j[t]]));
#pragma unroll
                                for (int q = 0; q < kQMax; ++q)
                                    if (q < Q) out = out && order_key(__dadd_ru(acc[t][q], W.scq[q])) < kr;
                            }
                            if (__all_sync(0xffffffffu, out)) {
                                all_out = true;
                                break;
                            }
                        }
                    }
                }
#pragma unroll
                for (int t = 0; t < TC; ++t) {
                    uint32_t b = 0, cb = 0;
#pragma unroll
                    for (int q = 0; q < kQMax; ++q) {
                        if (!all_out && q < Q && ge_threshold(acc[t][q], to[t])) b |= 1u << q;
                        if (!all_out && q < Q && ge_threshold(acc[t][q], ti[t])) cb |= 1u << q;
                    }
                    bits[t] = b;
                    cbits[t] = cb;
                }
            }
#pragma unroll
            for (int t = 0; t < TC; ++t) {
                bits[t] &= tri_mask[t];
                cbits[t] &= tri_mask[t];
            }
            if constexpr (!EMIT) {
                emit_direct<TC>(st, P, W.cperm, W.cmir, S.qid, R, I, lane, j, bits, cbits, rechecked);
            } else {
            // with distances every maybe-in pair is re-decided in binary64: the
            // pairs are compacted with one warp scan per half of the queries and
            // queued 32 at a time
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
            const uint32_t hm = half ? 0xFF00u : 0x00FFu;
            int cnt = 0;
#pragma unroll
            for (int t = 0; t < TC; ++t) cnt += __popc(bits[t] & hm);
            int total;
            int off = warp_excl_scan(cnt, lane, &total);
            if (total == 0) continue;
#pragma unroll
            for (int t = 0; t < TC; ++t) {
                uint32_t b = bits[t] & hm;
                while (b) {
                    const int q = __ffs(b) - 1;
                    b &= b - 1u;
                    W.list[off++] = (uint16_t)(((t * 32 + lane) << 4) | q);
                }
            }
            __syncwarp();
            for (int e0 = 0; e0 < total; e0 += 32) {
                const int e = e0 + lane;
                int nout = 0;
                int32_t qid = 0, cid = 0;
                double dist = 0.0;
                bool band = false, mir = false;
                int q = 0;
                int64_t jj = 0;
                if (e < total) {
                    const int ent = W.list[e];
                    const int slot = (ent >> 4) & 0x7FF;
                    q = ent & 15;
                    jj = W.cj[slot];
                    const int fl = W.cmir[slot];
                    mir = fl == 1 || (fl == 2 && jj != (int64_t)(I.q0 + q));
                    band = true;
                }
                const bool queued = band_push_q(bq, P, lane, band, I.q0 + q, (int32_t)jj, mir);
                if (band && !queued) {  // queue full: decide here
                    const double s = direct_sq(P.xs + (int64_t)(I.q0 + q) * DP, P.xs + jj * DP, P.d);
                    ++rechecked;
                    if (s <= R.e2) {
                        nout = mir ? 2 : 1;
                        qid = (int32_t)(S.qid[q] - R.off);
                        cid = (int32_t)(W.cperm[(W.list[e] >> 4) & 0x7FF] - R.off);
                        dist = sqrt(s);
                    }
                }
                stage_emit(st, P, lane, nout, qid, cid, dist);
            }
            __syncwarp();
            }
            }
            if constexpr (PRUNE) {
                head = (head + ns) & (CcWarpSmem<T, DP, TC, EMIT, RUNS, true>::RING - 1u);
                cnt -= ns;
                __syncwarp();
            } else {
                base += (uint32_t)SLOTS;
            }
        }
        __syncwarp();
    }
    band_q_close(bq, P, lane);
    stage_flush(st, P, lane);
    if (PRUNE && lane == 0 && W.pruned) atomicAdd(&P.counters[6], W.pruned);
    for (int o = 16; o > 0; o >>= 1) rechecked += __shfl_down_sync(0xffffffffu, rechecked, o);
    if (lane == 0 && rechecked) atomicAdd(&P.counters[2], rechecked);
}

// Whether a join's candidates pass the bounding-box prune: where items have more
// than 140 candidates, so that it saves whole chunks (of 128 candidates in FP64,
// 64 in FP32) and not slots of one, and in FP64 more than 300 evaluations, for
// its own cost an item; in FP64 with few items, which leave the chip waiting for
// single ones, above 90 (30,000 x 3-D, 110 candidates: 67.8 / 63.8).  Planar cells
// keep 83% of their candidates, so padded d = 2 goes without it in FP64 and above
// 70 candidates with it in FP32; joins without an index go without (the box of 16
// arbitrary points spans everything), and batches (no radius per instance for the
// FP64 tile).  Tile times without / with it, us, by candidates an item (200,000
// points): FP64 3-D 75 196 / 233, 150 362 / 273, 718 1183 / 1000; 4-D 24 252 /
// 325, 94 219 / 271, 175 337 / 267, 644 1028 / 717; 6-D 50 572 / 788, 149 (200
// evaluations) 862 / 960, 265 (440) 1108 / 1025, 2026 6070 / 2547; clusters 4-D
// 94 303 / 320, 295 664 / 578; 2-D 18 123 / 140, 355 626 / 625; 8-D without an
// index 6468 / 7373.  FP64 with distances 4-D 24 263 / 412, 175 335 / 289.  FP32
// with distances 3-D 39 91 / 102, 75 103 / 104, 150 150 / 144; 4-D 24 115 / 153,
// 94 99 / 106, 175 102 / 99, 644 204 / 176; 6-D 50 296 / 334, 149 474 / 428,
// 2026 766 / 565; 2-D 10 83 / 91, 37 115 / 115, 76 206 / 197, clusters 74 245 / 231.
inline bool cc_prune(const Index* ix, const JoinParams& p, bool fp64) {
    if (p.batch || ix->m == 0 || ix->n_cells <= 0) return false;
    const double n = (double)ix->n, ev = (double)ix->n_evaluated, items = (double)ix->n_cells + n / kQMax;
    if (ix->dp == 2) return !fp64 && ev > 70.0 * n;
    if (fp64 && items < 8192.0) return ev > 90.0 * n && ev > 300.0 * items;
    return ev > 140.0 * n && (!fp64 || ev > 300.0 * items);
}

template <typename T, int DP, bool EMIT, int RUNS, bool PRUNE>
inline int launch_dper(Index* ix, const JoinParams& p) {
    constexpr int TC = DP > 8 ? 2 : std::is_same<T, float>::value ? SJ_CC_TC_SMALL_D : 4;
    constexpr int NW = cc_warps<CcWarpSmem<T, DP, TC, EMIT, RUNS, PRUNE>>();
    auto kern = k_join_cc<T, DP, TC, EMIT, NW, RUNS, PRUNE>;
    int per_sm = 0;
    SJ_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, 0));
    if (per_sm < 1) per_sm = 1;
    long long blocks = (long long)device_sm_count(ix->device) * per_sm;
    const long long need = (ix->n_items + NW - 1) / NW;
    if (blocks > need) blocks = need > 0 ? need : 1;
    kern<<<(unsigned)blocks, NW * 32, 0, ix->stream>>>(p);
    note_launch();
    SJ_CK(cudaGetLastError());
    return SJ_OK;
}

// Run capacity of the item image: 3^(m-1) + 1 runs for m indexed dims; a
// grid of at most 4 dims needs 28, which keeps the per-warp shared memory of
// the small-d kernels small enough for 8 CTAs per SM.  Large-d kernels are
// bound by registers, so they keep the general capacity only.
template <typename T, int DP, bool EMIT>
inline int launch_dpe(Index* ix, const JoinParams& p) {
    if constexpr (DP <= 8) {
        if constexpr (DP > 2 || std::is_same<T, float>::value)
            if (cc_prune(ix, p, std::is_same<T, double>::value))
                return ix->m <= 4 ? launch_dper<T, DP, EMIT, 28, true>(ix, p)
                                  : launch_dper<T, DP, EMIT, kMaxRuns, true>(ix, p);
        return ix->m <= 4 ? launch_dper<T, DP, EMIT, 28, false>(ix, p) : launch_dper<T, DP, EMIT, kMaxRuns, false>(ix, p);
    } else {
        return launch_dper<T, DP, EMIT, kMaxRuns, false>(ix, p);
    }
}

// The tile launch for padded dimension DP.  The FP32 filter at DP <= 8
// without distances runs k_join_f32s (sj_join_f32s.cu) instead.
template <typename T, int DP>
int launch_cc_dp(Index* ix, const JoinParams& p) {
    if constexpr (std::is_same<T, float>::value && DP <= 8) {
        if (!p.emit_dist) {
            set_error("the FP32 filter at padded dimension %d without distances runs k_join_f32s", DP);
            return SJ_ERR_UNSUPPORTED;
        }
        return launch_dpe<T, DP, true>(ix, p);
    } else {
        return p.emit_dist ? launch_dpe<T, DP, true>(ix, p) : launch_dpe<T, DP, false>(ix, p);
    }
}


}  // namespace sj
