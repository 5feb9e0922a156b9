// Certified low-precision filter on the 5th-generation tensor cores
// (tcgen05.mma kind::f16, bf16 or fp16 operands, FP32 accumulation in TMEM).
//
// The dot products of Eq. 3 (the tensor-core part of Eq. 4) are formed from a
// bf16 split of every FP32 kernel coordinate, y = y1 + y2 + y3 exactly (8
// significant bits each).  BF16x3 keeps the six products whose term indices
// sum to at most 4: for dim k the candidate row holds (c1, c2, c1, c3, c2, c1)
// and the query row (q1, q1, q2, q1, q2, q3); BF16x2 keeps three, (c1, c2, c1)
// against (q1, q1, q2), for half the K; FP16x2 keeps the same three products
// of fp16 terms (11 significant bits) of the coordinates scaled by a power of
// two into fp16's range, for a narrower band.  Three more K slots carry the
// query's -||y_q||^2 / 2, split the same way, against ones, so the
// accumulator ends as a = -||y_q||^2/2 + y_q . y_c, the quantity every other
// kernel computes.  Each value is compared with per-candidate thresholds
// widened for this arithmetic (dropped split products and the tensor core's
// FP32 accumulation); what is maybe in goes, with what is certainly in, as
// records (a candidate against 32 query columns) to k_resolve, which decides
// the pairs inside the bound and writes the result (sj_resolve.cu).
//
// One persistent CTA per SM, warp-specialised:
//   warp 0      tiles: takes work items from the queue and cuts the item's
//               candidate runs into tiles (128 rows = 16 8-row groups), per
//               tile the rows' ranges and the copies that bring them, two
//               tiles at a time;
//   warp 1      MMA issuer (one thread): K/16 MMAs per tile into one of two
//               TMEM accumulators (128 lanes x N columns), committed to the
//               stage and accumulator barriers;
//   warp 2      copies (one thread): the item's query tile (MMA B, N <= 256
//               queries, 8-row groups from an 8-aligned start; the next
//               item's while this one runs, where shared memory allows) and
//               the candidate tiles (MMA A) in K-slices of 64, one or two a
//               pipeline stage, bulk copies completing on mbarriers;
//   warp 3      rows: position, flag and thresholds of the tile's rows, fetched
//               a tile ahead, into shared memory beside the accumulator;
//   warps 4..   epilogue (16 warps): each thread owns one candidate row (its
//               TMEM lane) and a quarter of its N accumulators (interleaved
//               32-column chunks): a max over the chunk against the row's
//               threshold first (hits are rare), then column masks of the
//               maybe-in and the certain ones and a record.
// What bounds it: at K = 208 the MMA (2.2 PFLOP/s of it when the epilogue is
// left out, 1.97 with it); at K = 64 the epilogue's instruction issue, so it holds
// only what has to happen while the accumulator is there, an accumulator is
// released as soon as its last columns are in registers, and a tile costs an
// epilogue warp one wait and one 16-byte read.  Each role's code is a short
// loop of its own: waits and copies of one thread cost some 250 cycles a stage
// beside 16 other warps, so serial work per slice, not bandwidth, kept the MMA
// waiting (one producer warp: 700 cycles a slice and up to 1,900 a tile of many
// runs; the 64-D workload was at half the MMA's rate with any number of stages,
// any copy size and half the MMAs left out).  Tile kernel with what follows it,
// at the outset / emission moved to k_resolve / roles split: 2^17 x 16-D without
// an index 2.93 / 2.06 / 1.71 ms, 500,000 x 16-D mixture 5.92 / 3.21 / 2.64,
// 200,000 x 64-D 8.09 / 7.10 / 4.15.  8 epilogue warps with two chunks in
// registers each instead of 16 with one: 2.40 / 3.48 / 2.83 (150,000 x 64-D,
// against 2.06 / 3.17 / 2.64).
// A symmetric join evaluates only the triangle of each self cell: the self
// run starts at the item's first query and pairs below the diagonal are
// masked.  Every wait is bounded; on expiry the CTA stops issuing work,
// drains its copies and MMAs (again bounded), frees TMEM and records an error
// the host reports as SJ_ERR_TIMEOUT.
#include <cuda_bf16.h>

#include "sj_join_common.cuh"

namespace sj {

constexpr int kTcM = 128;             // candidate rows per tile (TMEM lanes)
constexpr int kTcG = kTcM / 8;        // 8-row groups per tile
constexpr int kKS = 64;               // K per pipeline slice
constexpr int kMetaDepth = 8;         // tiles of row metadata in flight
constexpr int kTcEpi = 16;            // epilogue warps, four per TMEM lane quarter, splitting the columns
constexpr int kTcThreads = 128 + 32 * kTcEpi;  // tile, MMA, copy and row warps, epilogue
constexpr long long kTcSpin = 1 << 22;  // bound on barrier polls per wait

struct TcParams {
    const __nv_bfloat16* rows_a;  // candidate role, slice-major 8-row groups (16-bit terms)
    const __nv_bfloat16* rows_b;  // query role, same layout
    long long nrows;              // rows per slice (packed points, padded)
    int* error;                   // set to 1 when a bounded wait expires
    uint32_t ab_bf16;             // 1: A and B are bf16, 0: both fp16
};

template <int KP>
struct TcShape {
    static constexpr int NMAX = tc_nmax(KP);
    static constexpr int SLICES = (KP + kKS - 1) / kKS;
    // K-slices of a pipeline stage: the copy and the MMA thread pay a wait and
    // an arrival (about 250 cycles) a stage, so two where a tile has several
    static constexpr int GS = SLICES > 1 ? 2 : 1;
    static constexpr int GROUPS = (SLICES + GS - 1) / GS;
    static constexpr int A_SLICE = kTcM * kKS * 2;  // bytes
    static constexpr int A_STAGE = GS * A_SLICE;
    static constexpr int slice_k(int sl) { return KP - sl * kKS < kKS ? KP - sl * kKS : kKS; }
    static constexpr int B_BYTES = NMAX * KP * 2;
    static constexpr int NB = KP <= 112 ? 2 : 1;  // query tiles in flight (as shared memory allows)
};

// Per-item information shared by the roles (a ring of two).
struct TcItem {
    long long it;      // work item, or -1: no more work
    int q0, q1;        // queries [q0, q1)
    int qa;            // 8-aligned first row of the query tile
    int ncol;          // MMA N: query-tile rows, a multiple of 16
    int ntiles;        // candidate tiles
};

// Per-tile row metadata: each 8-row group's first row (-8: none), the run's
// valid position range and its flag (0 plain, 1 mirror, 2 self triangle); and
// the copies that bring the tile: rows of consecutive groups of the index.
struct TcMeta {
    int4 g[kTcG];       // first row, first and past-the-last valid position, flag
    int32_t nseg, cnt;  // copies, groups
    int4 seg[kTcG];     // first group in the tile, groups, first group of the index, -
};

template <int KP>
struct TcSmem {
    static constexpr int EPI = kTcEpi;
    static_assert(EPI % 4 == 0, "epilogue warps come in whole warpgroups");
    static constexpr int MAX_STAGES = 8;
    uint64_t a_full[MAX_STAGES], a_empty[MAX_STAGES];
    uint64_t b_full[2], b_empty[2];
    uint64_t item_full[2], item_empty[2];
    uint64_t meta_full[kMetaDepth], meta_empty[kMetaDepth];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t drain;
    uint32_t tmem;
    int abort;
    TcItem items[2];
    TcMeta meta[kMetaDepth];
    // per accumulator, what its epilogue needs of each row: candidate position,
    // flag, and the negated thresholds as floats (-inf: no candidate)
    int4 rows[2][kTcM];
    int32_t rgp[kMaxRuns];  // tile warp: per run of the item, its first group's number in the item
    int32_t rlo[kMaxRuns], rhi[kMaxRuns];
    uint8_t rfl[kMaxRuns];
};

// Operand stages: as many as fit (up to 8) in the 227 KB of shared memory a
// CTA may use next to the query tile and the rest.
constexpr size_t kSmemMax = 232448;
template <int KP>
__host__ __device__ constexpr int tc_stages() {
    const long long left = (long long)kSmemMax - 1024 - TcShape<KP>::NB * TcShape<KP>::B_BYTES - (long long)sizeof(TcSmem<KP>);
    const long long st = left / TcShape<KP>::A_STAGE;
    return st > TcSmem<KP>::MAX_STAGES ? TcSmem<KP>::MAX_STAGES : (int)st;
}
template <int KP>
constexpr size_t tc_smem_bytes() {
    return 1024 /* alignment slack */ + (size_t)TcShape<KP>::NB * TcShape<KP>::B_BYTES +
           (size_t)tc_stages<KP>() * TcShape<KP>::A_STAGE + sizeof(TcSmem<KP>);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major core matrices (8 rows x 16 bytes,
// contiguous along K), 8-row groups `sbo` bytes apart, no swizzle; a K step of 16
// advances the address by 256 bytes.  (The 128-byte swizzled layout ran at the
// same speed: 2.38 / 2.34 ms for 150,000 x 64-D.)
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(128 >> 4) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version bits 46-48 = 0b001
    return d;
}

// Instruction descriptor of kind::f16: D f32, A and B of one type (bf16 when
// ab_bf16 = 1, else fp16), both K-major.
__host__ __device__ constexpr uint32_t umma_idesc(int m, int n, uint32_t ab_bf16) {
    return (1u << 4) | ((ab_bf16 & 1u) << 7) | ((ab_bf16 & 1u) << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

// One lane of a converged warp (the compiler then knows that one thread runs
// the branch, and keeps the operands of copies and MMAs in uniform registers).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}" : "=r"(p));
    return p != 0u;
}
__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void bar_arrive_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(smem_u32(b)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool bar_test(uint64_t* b, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return done != 0;
}
// Waits for the phase of the given parity; false when the CTA aborts or the
// bound (polls) expires, which raises the abort.
__device__ __forceinline__ bool bar_wait_n(uint64_t* b, uint32_t parity, volatile int* abort, long long polls) {
    for (long long i = 0; i < polls; ++i) {
        if (bar_test(b, parity)) return true;
        if (*abort) return false;
    }
    *abort = 1;
    return false;
}
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity, volatile int* abort) {
    return bar_wait_n(b, parity, abort, kTcSpin);
}
// The wait of a whole warp: one answer for all lanes.
__device__ __forceinline__ bool bar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort) {
    return __all_sync(0xffffffffu, bar_wait(b, parity, abort));
}
// Bulk copy global -> shared completing on an mbarrier.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// Three-input maximum (one instruction on this architecture).
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// (mask << 1) | sign bit of v: one funnel shift.
__device__ __forceinline__ uint32_t push_sign(uint32_t mask, float v) {
    return __funnelshift_l(__float_as_uint(v), mask, 1);
}

// 32 consecutive TMEM columns of this thread's lane (no wait).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
}

// A record: one candidate against 32 query positions from a first one on, as
// (maybe-in columns, certain ones, first position, candidate position | kMirrorBit
// when its pairs are emitted in both orders, the diagonal excepted).  A warp
// takes room in the queue 64 records at a time with one atomic.
constexpr int kTcChunk = 64;
struct TcRecords {
    unsigned long long base;  // next reserved record
    int left;                 // reserved records left (warp-uniform)
    bool over;                // the reservation goes past the queue
};

// Squared distance of two kernel-coordinate rows in binary32, rows of dp floats
// (resolve's refine_sq, for a padded dimension known at run time).
__device__ __forceinline__ float tc_refine_sq(const float* __restrict__ a, const float* __restrict__ b, int dp) {
    float s = 0.f;
    for (int k = 0; k < dp; k += 2) {
        const float2 u = *reinterpret_cast<const float2*>(a + k), v = *reinterpret_cast<const float2*>(b + k);
        const float t0 = u.x - v.x, t1 = u.y - v.y;
        s = __fmaf_rn(t0, t0, s);
        s = __fmaf_rn(t1, t1, s);
    }
    return s;
}

// Warp-collective: records that found no room in the queue (queue_entries; no
// columns: none of this lane), all of one item.  Their pairs are decided as in k_resolve and written here:
// without distances the uncertain columns first, then one reservation for all
// pairs of the warp's records, a column of every lane at a time (one position
// after another: the writes are coalesced); with distances, whose binary64 sums
// are then needed once, a reservation per column.  Measured, 2^17 x 16-D without
// an index, 5,800 neighbours (759 M pairs, about half of the records past the
// queue): 10.8 ms, clustered 11.9 (before there were records 13.8 and 13.7; each
// lane on its own, every pair in binary64 with an atomic of its own, 79 and 109).
__device__ __noinline__ void tc_resolve_here(const JoinParams& P, int lane, int4 e) {
    const unsigned some = __ballot_sync(0xffffffffu, e.x != 0), lt = (1u << lane) - 1u;
    if (some == 0u) return;
    const int32_t cs = (int32_t)((uint32_t)e.w & ~kMirrorBit);
    const bool mirrored = e.w < 0;
    double e2 = P.e2;
    float2 r = make_float2(P.refine_out, P.refine_in);
    int gid = 0;
    int32_t off = 0;
    unsigned long long* cursor = &P.counters[1];
    if (P.batch) {
        const int li = P.batch->inst_of_sorted[__shfl_sync(0xffffffffu, cs, __ffs(some) - 1)];
        e2 = P.batch->inst_e2[li];
        r = P.batch->inst_refine[li];
        gid = P.batch->inst_gid[li];
        off = (int32_t)P.batch->inst_off[li];
        cursor = &P.batch->cursor[gid];
    }
    const float* __restrict__ Y = static_cast<const float*>(P.y);
    const bool dist = P.emit_dist != 0;
    uint32_t left = (uint32_t)e.x;
    const uint32_t open = dist ? left : left & ~(uint32_t)e.y;
    const unsigned decided = __reduce_add_sync(0xffffffffu, (unsigned)__popc(open));
    if (lane == 0 && decided) atomicAdd(&P.counters[2], (unsigned long long)decided);
    const int32_t cid = e.x != 0 ? P.perm[cs] - off : 0;
    unsigned long long at = 0;
    if (!dist) {
        for (uint32_t m = open; m; m &= m - 1u) {
            const int32_t qs = e.z + __ffs(m) - 1;
            const float s32 = tc_refine_sq(Y + (int64_t)qs * P.dp, Y + (int64_t)cs * P.dp, P.dp);
            const bool in = s32 < r.y || (!(s32 > r.x) && direct_sq(P.xs + (int64_t)qs * P.dp,
                                                                    P.xs + (int64_t)cs * P.dp, P.d) <= e2);
            if (!in) left &= ~(m & (0u - m));
        }
        unsigned nout = (unsigned)__popc(left) << (mirrored ? 1 : 0);
        const int diag = cs - e.z;
        if (mirrored && diag >= 0 && diag < 32 && (left >> diag & 1u)) --nout;
        const unsigned total = __reduce_add_sync(0xffffffffu, nout);
        if (total == 0u) return;
        if (lane == 0) at = atomicAdd(cursor, (unsigned long long)total);
        at = __shfl_sync(0xffffffffu, at, 0);
    }
    while (__any_sync(0xffffffffu, left != 0u)) {
        bool has = left != 0u;
        const int32_t qs = has ? e.z + __ffs(left) - 1 : 0;
        left &= left - 1u;
        double s = 0.0;
        if (dist && has) {
            s = direct_sq(P.xs + (int64_t)qs * P.dp, P.xs + (int64_t)cs * P.dp, P.d);
            has = s <= e2;
            s = sqrt(s);
        }
        const bool two = has && mirrored && cs != qs;
        const unsigned b1 = __ballot_sync(0xffffffffu, has), b2 = __ballot_sync(0xffffffffu, two);
        const unsigned n = (unsigned)(__popc(b1) + __popc(b2));
        if (dist && n > 0u) {
            if (lane == 0) at = atomicAdd(cursor, (unsigned long long)n);
            at = __shfl_sync(0xffffffffu, at, 0);
        }
        if (has) {
            const int32_t qid = P.perm[qs] - off;
            const unsigned long long p = at + (unsigned long long)(__popc(b1 & lt) + __popc(b2 & lt));
            for (int u = 0; u < (two ? 2 : 1); ++u) {
                const int2 pair = u == 0 ? make_int2(qid, cid) : make_int2(cid, qid);
                if (P.batch) {
                    const long long slot = batch_slot(*P.batch, gid, p + (unsigned)u);
                    if (slot >= 0) {
                        P.batch->pool[slot] = pair;
                        if (dist) P.batch->dpool[slot] = s;
                    }
                } else if (p + (unsigned)u < P.capacity) {
                    P.out_pairs[p + (unsigned)u] = pair;
                    if (dist) P.out_dist[p + (unsigned)u] = s;
                }
            }
        }
        at += n;
    }
}

// Warp-collective: the lanes whose record has columns append it.
__device__ __forceinline__ void tc_record(TcRecords& rec, const JoinParams& P, int lane, int4 e) {
    const unsigned b = __ballot_sync(0xffffffffu, e.x != 0);
    const int n = __popc(b), r = __popc(b & ((1u << lane) - 1u));
    unsigned long long pos = rec.base + (unsigned long long)r;
    if (n <= rec.left) {
        rec.base += (unsigned long long)n;
        rec.left -= n;
    } else {  // the rest of this reservation, then a fresh one (n <= 32 < kTcChunk)
        unsigned long long fresh = 0;
        if (lane == 0) fresh = atomicAdd(&P.counters[3], (unsigned long long)kTcChunk);
        fresh = __shfl_sync(0xffffffffu, fresh, 0);
        if (r >= rec.left) pos = fresh + (unsigned long long)(r - rec.left);
        const int used = n - rec.left;
        rec.base = fresh + (unsigned long long)used;
        rec.left = kTcChunk - used;
        rec.over = fresh + kTcChunk > P.band_cap >> 1;
    }
    const bool fits = pos < P.band_cap >> 1;
    if (e.x != 0 && fits) reinterpret_cast<int4*>(P.band)[pos] = e;
    if (rec.over) tc_resolve_here(P, lane, fits ? make_int4(0, 0, 0, 0) : e);  // (uniform)
}

// DBG: the recording instantiation of the filter dump (a test aid; the join
// kernels proper carry none of its code).
template <int KP, bool DBG>
__global__ void __launch_bounds__(kTcThreads, 1) k_join_tc(JoinParams P, TcParams T) {
    using SH = TcShape<KP>;
    using SM = TcSmem<KP>;
    constexpr int STAGES = tc_stages<KP>();
    static_assert(STAGES >= 2, "at least two operand stages");
    static_assert(kTcG == 16, "the tile warp resolves two tiles of 16 groups at a time");
    constexpr int NMAX = SH::NMAX;
    extern __shared__ unsigned char dsm_raw[];
    unsigned char* dsm = reinterpret_cast<unsigned char*>(((uintptr_t)dsm_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sB = dsm;
    unsigned char* sA = dsm + SH::NB * SH::B_BYTES;
    SM& S = *reinterpret_cast<SM*>(sA + (size_t)STAGES * SH::A_STAGE);
    volatile int* abort = &S.abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            bar_init(&S.a_full[i], 1);
            bar_init(&S.a_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(&S.b_full[i], 1);
            bar_init(&S.b_empty[i], 1);
            bar_init(&S.item_full[i], 1);
            bar_init(&S.item_empty[i], 3 + SM::EPI);  // the MMA and copy threads, the row and epilogue warps
            bar_init(&S.acc_full[i], 2);              // the MMAs are done, the rows written
            bar_init(&S.acc_empty[i], SM::EPI);
        }
        for (int i = 0; i < kMetaDepth; ++i) {
            bar_init(&S.meta_full[i], 1);
            bar_init(&S.meta_empty[i], 2);  // the copy thread and the row warp
        }
        bar_init(&S.drain, 1);
        S.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"((uint32_t)(2 * NMAX)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = S.tmem;

    if (warp == 0) {
        // ------------------------------------------------------------ tiles
        // Takes the work items and cuts their candidates into tiles: lane i
        // of a tile resolves the tile's 8-row group i (a binary search over
        // the item's per-run group prefix); runs of consecutive groups become
        // one copy each.  Runs ahead of the copies by the depth of the
        // metadata ring.
        uint32_t m_i = 0, m_ph = 0, it_i = 0, it_ph = 0;
        for (;;) {
            long long it = 0;
            if (lane == 0) it = (long long)atomicAdd(&P.counters[0], 1ull);
            it = __shfl_sync(0xffffffffu, it, 0);
            Item I{0, 0, 0, 0};
            if (it < P.n_items) I = P.items[it];
            const int nr = it < P.n_items ? I.r1 - I.r0 : 0;
            // per run: first group, valid range, flag and the exclusive group prefix
            int carry = 0;
            for (int r0 = 0; r0 < nr; r0 += 32) {
                const int r = r0 + lane;
                int cnt = 0;
                if (r < nr) {
                    const Run R = P.runs[I.r0 + r];
                    const bool mir = (R.end_flags & kMirrorBit) != 0;
                    const bool self = P.tri && !mir;
                    const int32_t lo = self ? I.q0 : R.start;
                    const int32_t hi = (int32_t)(R.end_flags & ~kMirrorBit);
                    cnt = hi > lo ? ((hi - 1) >> 3) - (lo >> 3) + 1 : 0;
                    S.rlo[r] = lo;
                    S.rhi[r] = hi;
                    S.rfl[r] = (uint8_t)(mir ? 1 : (self ? 2 : 0));
                }
                int x = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (r < nr) S.rgp[r] = carry + x - cnt;
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
            const int ngroups = carry;
            __syncwarp();
            const int ntiles = (ngroups + kTcG - 1) / kTcG;
            // the ring slot is free once its previous item is done
            if (!bar_wait_warp(&S.item_empty[it_i], it_ph ^ 1u, abort)) break;
            if (lane == 0) {
                TcItem& X = S.items[it_i];
                X.it = it < P.n_items ? it : -1;
                X.q0 = I.q0;
                X.q1 = I.q1;
                X.qa = I.q0 & ~7;
                X.ncol = ((I.q1 - X.qa) + 15) & ~15;
                X.ntiles = ntiles;
                bar_arrive(&S.item_full[it_i]);
            }
            if (it >= P.n_items) break;
            if (++it_i == 2) it_i = 0, it_ph ^= 1u;
            bool bail = false;
            for (int t0 = 0; t0 < ntiles && !bail; t0 += 2) {
                // this lane's group, of tile t0 (lanes 0 .. 15) or t0 + 1
                const int j = t0 * kTcG + lane;
                int4 g = make_int4(-8, 0, 0, 0);
                if (j < ngroups) {
                    int lo = 0, hi = nr - 1;  // last run whose prefix is <= j
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (S.rgp[mid] <= j)
                            lo = mid;
                        else
                            hi = mid - 1;
                    }
                    g = make_int4((S.rlo[lo] & ~7) + 8 * (j - S.rgp[lo]), S.rlo[lo], S.rhi[lo], S.rfl[lo]);
                }
                // runs of consecutive groups in a tile: their first lanes
                const int32_t gprev = __shfl_up_sync(0xffffffffu, g.x, 1);
                const bool first = j < ngroups && ((lane & (kTcG - 1)) == 0 || g.x != gprev + 8);
                const uint32_t firsts = __ballot_sync(0xffffffffu, first);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (t0 + u >= ntiles) break;
                    const int cnt = min(ngroups - (t0 + u) * kTcG, kTcG), l = lane - u * kTcG;
                    const uint32_t mine = (firsts >> (u * kTcG)) & 0xFFFFu;
                    if (!bar_wait_warp(&S.meta_empty[m_i], m_ph ^ 1u, abort)) {
                        bail = true;
                        break;
                    }
                    TcMeta& M = S.meta[m_i];
                    if (l >= 0 && l < kTcG) {
                        M.g[l] = g;
                        if (first) {
                            const uint32_t later = mine & ~((2u << l) - 1u);
                            M.seg[__popc(mine & ((1u << l) - 1u))] =
                                make_int4(l, (later ? __ffs(later) - 1 : cnt) - l, g.x >> 3, 0);
                        }
                    }
                    if (lane == 0) {
                        M.nseg = __popc(mine);
                        M.cnt = cnt;
                    }
                    __syncwarp();
                    if (lane == 0) bar_arrive(&S.meta_full[m_i]);
                    if (++m_i == kMetaDepth) m_i = 0, m_ph ^= 1u;
                }
            }
            if (bail) break;
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ copies
        // One thread: per item the query tile, per tile and K-slice one bulk
        // copy for each run of consecutive groups.
        if (elect_one()) {
            uint32_t a_i = 0, a_ph = 0, m_i = 0, m_ph = 0, it_i = 0, it_ph = 0, b_i = 0, b_ph = 0;
            // stages and query tiles armed so far, and the parity of the last arming
            uint32_t armed_a = 0, par_a = 0, armed_b = 0, par_b = 0;
            bool bail = false;
            while (!bail) {
                if (!bar_wait(&S.item_full[it_i], it_ph, abort)) break;
                const TcItem X = S.items[it_i];
                bar_arrive(&S.item_empty[it_i]);
                if (X.it < 0) break;
                if (++it_i == 2) it_i = 0, it_ph ^= 1u;
                // the query tile, one copy per K-slice
                if (!bar_wait(&S.b_empty[b_i], b_ph ^ 1u, abort)) break;
                const uint32_t gq = (uint32_t)(X.ncol >> 3);
                bar_arrive_tx(&S.b_full[b_i], gq * KP * 16u);
                armed_b |= 1u << b_i;
                par_b = (par_b & ~(1u << b_i)) | (b_ph << b_i);
                for (int sl = 0; sl < SH::SLICES; ++sl) {
                    const int ks = KP - sl * kKS < kKS ? KP - sl * kKS : kKS;
                    const __nv_bfloat16* src =
                        T.rows_b + (long long)sl * kKS * T.nrows + (long long)(X.qa >> 3) * ks * 8;
                    bulk_g2s(smem_u32(sB) + b_i * (uint32_t)SH::B_BYTES + (uint32_t)(NMAX * 2 * kKS * sl), src,
                             gq * (uint32_t)ks * 16u, smem_u32(&S.b_full[b_i]));
                }
                if (++b_i == SH::NB) b_i = 0, b_ph ^= 1u;
                for (int t = 0; t < X.ntiles && !bail; ++t) {
                    if (!bar_wait(&S.meta_full[m_i], m_ph, abort)) {
                        bail = true;
                        break;
                    }
                    const TcMeta& M = S.meta[m_i];
                    const int nseg = M.nseg, cnt = M.cnt;
#pragma unroll 1
                    for (int g = 0; g < SH::GROUPS; ++g) {
                        if (!bar_wait(&S.a_empty[a_i], a_ph ^ 1u, abort)) {
                            bail = true;
                            break;
                        }
                        const int k0 = g * SH::GS * kKS, gk = KP - k0 < SH::GS * kKS ? KP - k0 : SH::GS * kKS;
                        bar_arrive_tx(&S.a_full[a_i], (uint32_t)(cnt * gk) * 16u);
                        armed_a |= 1u << a_i;
                        par_a = (par_a & ~(1u << a_i)) | (a_ph << a_i);
                        const uint32_t dst = smem_u32(sA) + a_i * (uint32_t)SH::A_STAGE, bar = smem_u32(&S.a_full[a_i]);
                        const char* src = reinterpret_cast<const char*>(T.rows_a) + 2 * k0 * T.nrows;
#pragma unroll 1
                        for (int k = 0; k < nseg; ++k) {
                            const int4 e = M.seg[k];
                            uint32_t to = dst;
                            const char* from = src;
#pragma unroll
                            for (int u = 0; u < SH::GS; ++u) {
                                const int left = gk - u * kKS, ks16 = (left < kKS ? left : kKS) * 16;  // bytes a group
                                if (left > 0)
                                    bulk_g2s(to + (uint32_t)(e.x * ks16), from + (long long)e.z * ks16,
                                             (uint32_t)(e.y * ks16), bar);
                                to += (uint32_t)SH::A_SLICE;
                                from += 2 * kKS * T.nrows;
                            }
                        }
                        if (++a_i == STAGES) a_i = 0, a_ph ^= 1u;
                    }
                    bar_arrive(&S.meta_empty[m_i]);
                    if (++m_i == kMetaDepth) m_i = 0, m_ph ^= 1u;
                }
            }
            if (*abort) {
                // drain the copies this CTA armed (bounded), so none lands after exit
                for (int i = 0; i < STAGES; ++i)
                    if (armed_a >> i & 1u)
                        for (long long k = 0; k < kTcSpin && !bar_test(&S.a_full[i], par_a >> i & 1u); ++k) {
                        }
                for (int i = 0; i < SH::NB; ++i)
                    if (armed_b >> i & 1u)
                        for (long long k = 0; k < kTcSpin && !bar_test(&S.b_full[i], par_b >> i & 1u); ++k) {
                        }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            uint32_t a_i = 0, a_ph = 0, it_i = 0, it_ph = 0, b_i = 0, b_ph = 0, acc = 0, acc_ph = 0;
            bool issued = false;
            for (;;) {
                if (!bar_wait(&S.item_full[it_i], it_ph, abort)) break;
                const TcItem X = S.items[it_i];
                if (X.it < 0) break;
                if (!bar_wait(&S.b_full[b_i], b_ph, abort)) break;
                const uint32_t idesc = umma_idesc(kTcM, X.ncol, T.ab_bf16);
                bool fail = false;
                for (int t = 0; t < X.ntiles && !fail; ++t) {
                    if (!bar_wait(&S.acc_empty[acc], acc_ph ^ 1u, abort)) {
                        fail = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t dt = tmem + acc * NMAX;
                    // (unrolled: the descriptors are an address and constants,
                    // so a K step is issued in a few cycles)
#pragma unroll
                    for (int g = 0; g < SH::GROUPS; ++g) {
                        if (!bar_wait(&S.a_full[a_i], a_ph, abort)) {
                            fail = true;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        const uint32_t a0 = smem_u32(sA) + a_i * (uint32_t)SH::A_STAGE;
                        const uint32_t b0 = smem_u32(sB) + b_i * (uint32_t)SH::B_BYTES;
#pragma unroll
                        for (int u = 0; u < SH::GS; ++u) {
                            const int sl = g * SH::GS + u;
                            if (sl >= SH::SLICES) break;
                            const int ks = SH::slice_k(sl);
                            const uint64_t ad = umma_desc(a0 + (uint32_t)(u * SH::A_SLICE), (uint32_t)ks * 16u);
                            const uint64_t bd = umma_desc(b0 + (uint32_t)(NMAX * 2 * kKS * sl), (uint32_t)ks * 16u);
#pragma unroll
                            for (int kk = 0; kk < ks / 16; ++kk) {
                                const uint32_t accum = (sl > 0 || kk > 0) ? 1u : 0u;
                                asm volatile(
                                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dt),
                                    "l"(ad + 16u * kk), "l"(bd + 16u * kk), "r"(idesc), "r"(accum));
                            }
                        }
                        issued = true;
                        umma_commit(&S.a_empty[a_i]);  // the stage is free once these MMAs are done
                        if (++a_i == STAGES) a_i = 0, a_ph ^= 1u;
                    }
                    if (fail) break;
                    umma_commit(&S.acc_full[acc]);
                    if (++acc == 2) acc = 0, acc_ph ^= 1u;
                }
                if (fail) break;
                umma_commit(&S.b_empty[b_i]);  // the query tile is free once this item's MMAs are done
                if (++b_i == SH::NB) b_i = 0, b_ph ^= 1u;
                bar_arrive(&S.item_empty[it_i]);
                if (++it_i == 2) it_i = 0, it_ph ^= 1u;
            }
            if (issued) {
                // every MMA of this CTA has completed before TMEM is freed
                umma_commit(&S.drain);
                for (long long k = 0; k < kTcSpin && !bar_test(&S.drain, 0); ++k) {
                }
            }
        }
    } else if (warp == 3) {
        // ------------------------------------------------------------ rows
        // Four rows a lane: position, flag and thresholds of the next tile are
        // fetched while the current one's are handed over, so that an epilogue
        // warp reads 16 bytes a row and nothing else.
        const float* __restrict__ TO = static_cast<const float*>(P.thr_out);
        const float* __restrict__ TI = static_cast<const float*>(P.thr_in);
        uint32_t it_i = 0, it_ph = 0, m_i = 0, m_ph = 0, acc = 0, acc_ph = 0;
        // (the loaded thresholds are first touched a tile later)
        int32_t np[4], nfl[4];  // position, flag (-1: no candidate)
        float nto[4], nti[4];
        auto fetch = [&]() -> bool {
            if (!bar_wait_warp(&S.meta_full[m_i], m_ph, abort)) return false;
            const TcMeta& M = S.meta[m_i];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int row = 32 * u + lane;
                const int4 g = M.g[row >> 3];
                np[u] = g.x + (row & 7);
                const bool valid = g.x >= 0 && np[u] >= g.y && np[u] < g.z &&
                                   SJ_BOUND(P, np[u] < P.n_points, 31);
                nfl[u] = valid ? g.w : -1;
                const int32_t pl = valid ? np[u] : 0;
                nto[u] = TO[pl];
                nti[u] = TI[pl];
            }
            __syncwarp();
            if (lane == 0) bar_arrive(&S.meta_empty[m_i]);
            if (++m_i == kMetaDepth) m_i = 0, m_ph ^= 1u;
            return true;
        };
        bool bail = false;
        while (!bail) {
            if (!bar_wait_warp(&S.item_full[it_i], it_ph, abort)) break;
            const long long it = S.items[it_i].it;
            const int ntiles = S.items[it_i].ntiles;
            __syncwarp();
            if (lane == 0) bar_arrive(&S.item_empty[it_i]);
            if (it < 0) break;
            if (++it_i == 2) it_i = 0, it_ph ^= 1u;
            if (ntiles > 0 && !fetch()) break;
            for (int t = 0; t < ntiles; ++t) {
                int4 now[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    // (negated, never -0: the sign of a round-to-nearest sum
                    // a + nto is that of the exact a - threshold)
                    now[u] = make_int4(np[u], nfl[u], nfl[u] >= 0 ? __float_as_int(__fsub_rn(0.f, nto[u])) : (int)0xFF800000u,
                                       nfl[u] >= 0 ? __float_as_int(__fsub_rn(0.f, nti[u])) : (int)0xFF800000u);
                if ((t + 1 < ntiles && !fetch()) || !bar_wait_warp(&S.acc_empty[acc], acc_ph ^ 1u, abort)) {
                    bail = true;
                    break;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) S.rows[acc][32 * u + lane] = now[u];
                __syncwarp();
                if (lane == 0) bar_arrive(&S.acc_full[acc]);
                if (++acc == 2) acc = 0, acc_ph ^= 1u;
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int ew = warp - 4;
        const int quarter = warp & 3;  // TMEM lanes 32 quarter .. + 31
        const int part = ew >> 2;      // 32-column chunks part, part + EPI / 4, ...
        constexpr int CSTEP = 32 * (SM::EPI / 4);
        TcRecords rec{0, 0, false};
        uint32_t it_i = 0, it_ph = 0, acc = 0, acc_ph = 0;
        for (;;) {
            if (!bar_wait_warp(&S.item_full[it_i], it_ph, abort)) break;
            const TcItem X = S.items[it_i];
            if (X.it < 0) break;
            bool fail = false;
            for (int t = 0; t < X.ntiles; ++t) {
                if (!bar_wait_warp(&S.acc_full[acc], acc_ph, abort)) {
                    fail = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                // this thread's candidate row
                const int4 row = S.rows[acc][quarter * 32 + lane];
                const int32_t cp = row.x;
                const float nto = __int_as_float(row.z), nti = __int_as_float(row.w);
                const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + acc * NMAX;
                // the accumulator is released as soon as this warp's last
                // columns are in registers, before they are looked at
                for (int c0 = 32 * part; c0 < X.ncol || c0 == 32 * part; c0 += CSTEP) {
                    // (whole chunks, no branch around the load: columns past the
                    // accumulated ones hold an earlier tile's and are left out below)
                    uint32_t v[32];
                    tmem_ld32(taddr + (uint32_t)c0, v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (X.ncol - c0 <= CSTEP) {  // (this warp's last chunk)
                        asm volatile("tcgen05.fence::before_thread_sync;");
                        __syncwarp();
                        if (lane == 0) bar_arrive(&S.acc_empty[acc]);
                        if (X.ncol <= c0) break;
                    }
                    // maxima of 8-column groups, then of all 32 (three-input max)
                    const float* f = reinterpret_cast<const float*>(v);
                    float m8[4];
#pragma unroll
                    for (int g8 = 0; g8 < 4; ++g8)
                        m8[g8] = max3f(max3f(f[8 * g8], f[8 * g8 + 1], f[8 * g8 + 2]),
                                       max3f(f[8 * g8 + 3], f[8 * g8 + 4], f[8 * g8 + 5]),
                                       fmaxf(f[8 * g8 + 6], f[8 * g8 + 7]));
                    if (X.ncol - c0 < 32) m8[2] = m8[3] = -INFINITY;  // (a 16-column tail)
                    const float top = max3f(m8[0], m8[1], fmaxf(m8[2], m8[3]));
                    if (!DBG && !__any_sync(0xffffffffu, __fadd_rn(top, nto) >= 0.f)) continue;
                    // this row's columns: the item's, and in a self-cell triangle
                    // those at or below the candidate
                    const int lo = max(X.q0 - X.qa - c0, 0);
                    const int hi = min((row.y == 2 ? min(X.q1 - 1, cp) : X.q1 - 1) - X.qa - c0, 31);
                    const uint32_t cols = lo <= hi && row.z != (int)0xFF800000u
                                              ? (0xFFFFFFFFu << lo) & (0xFFFFFFFFu >> (31 - hi)) : 0u;
                    if (DBG) {  // the filter dump (test aid; constant indices: v stays in registers)
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (cols >> k & 1u) dbg_record(P, X.qa + c0 + k, cp, f[k]);
                    }
                    // bit k: column c0 + k is maybe in / certainly in
                    uint32_t mo = 0u, mi = 0u;
#pragma unroll
                    for (int g8 = 0; g8 < 4; ++g8) {
                        if (!__any_sync(0xffffffffu, __fadd_rn(m8[g8], nto) >= 0.f)) continue;
                        // sign of a - threshold: a miss
                        uint32_t no = 0u, ni = 0u;
#pragma unroll
                        for (int k = 6; k >= 0; k -= 2) {
                            const float2 a = make_float2(f[8 * g8 + k], f[8 * g8 + k + 1]);
                            const float2 o = __fadd2_rn(a, make_float2(nto, nto));
                            const float2 n = __fadd2_rn(a, make_float2(nti, nti));
                            no = push_sign(push_sign(no, o.y), o.x);
                            ni = push_sign(push_sign(ni, n.y), n.x);
                        }
                        mo |= (~no & 0xFFu) << (8 * g8);
                        mi |= (~ni & 0xFFu) << (8 * g8);
                    }
                    tc_record(rec, P, lane, make_int4((int)(mo & cols), (int)mi, X.qa + c0,
                                                      (int)((uint32_t)cp | (row.y ? kMirrorBit : 0u))));
                }
                if (++acc == 2) acc = 0, acc_ph ^= 1u;
            }
            if (fail) break;
            __syncwarp();
            if (lane == 0) bar_arrive(&S.item_empty[it_i]);
            if (++it_i == 2) it_i = 0, it_ph ^= 1u;
        }
        // the warp's unfilled records are closed (no columns)
        for (int i = lane; i < rec.left; i += 32)
            if (rec.base + (unsigned long long)i < (P.band_cap >> 1))
                reinterpret_cast<int4*>(P.band)[rec.base + (unsigned long long)i] = make_int4(0, 0, 0, 0);
    }

    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (tid == 0 && S.abort) atomicExch(T.error, 1);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * NMAX)));
    }
}

// Self-test of the bounded waits: one thread waits on an mbarrier that
// nothing arrives on; the wait must give up after its bound and raise the
// abort flag.  out[0] = 1 when the wait gave up, out[1] = the abort flag.
__global__ void k_wait_selftest(int* out, long long polls) {
    __shared__ uint64_t bar;
    __shared__ int abort;
    if (threadIdx.x == 0) {
        bar_init(&bar, 1);
        abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool done = bar_wait_n(&bar, 0, &abort, polls);
        out[0] = done ? 0 : 1;
        out[1] = abort;
    }
}

int selftest_bounded_wait(cudaStream_t s) {
    int* d = nullptr;
    SJ_TRY(dev_alloc_t(&d, 2, s));
    SJ_CK(cudaMemsetAsync(d, 0, 2 * sizeof(int), s));
    k_wait_selftest<<<1, 32, 0, s>>>(d, 1 << 16);
    note_launch();
    SJ_CK(cudaGetLastError());
    int h[2] = {0, 0};
    SJ_CK(cudaMemcpyAsync(h, d, sizeof h, cudaMemcpyDeviceToHost, s));
    SJ_CK(cudaStreamSynchronize(s));
    dev_free(d, s);
    if (h[0] == 1 && h[1] == 1) {
        set_error("the bounded wait gave up as designed");
        return SJ_ERR_TIMEOUT;
    }
    set_error("the bounded wait did not give up (%d, %d)", h[0], h[1]);
    return SJ_ERR_CUDA;
}

template <int KP, bool DBG>
static int launch_kp(Index* ix, const JoinParams& p, const TcParams& t) {
    auto kern = k_join_tc<KP, DBG>;
    const size_t smem = tc_smem_bytes<KP>();
    if (smem > kSmemMax) {
        set_error("tensor-core tile does not fit in shared memory (K = %d)", KP);
        return SJ_ERR_UNSUPPORTED;
    }
    SJ_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    constexpr int threads = kTcThreads;
    SJ_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) {
        set_error("tensor-core tile does not fit on an SM (K = %d)", KP);
        return SJ_ERR_UNSUPPORTED;
    }
    // one CTA per SM: it holds up to all 512 TMEM columns
    long long blocks = (long long)device_sm_count(ix->device);
    if (blocks > ix->n_items) blocks = ix->n_items > 0 ? ix->n_items : 1;
    kern<<<(unsigned)blocks, threads, smem, ix->stream>>>(p, t);
    note_launch();
    SJ_CK(cudaGetLastError());
    return SJ_OK;
}

template <int KP>
static int launch_k(Index* ix, const JoinParams& p, const TcParams& t) {
    return p.dbg ? launch_kp<KP, true>(ix, p, t) : launch_kp<KP, false>(ix, p, t);  // (dbg: the filter dump)
}

int launch_join_tc(Index* ix, const JoinOut& out, int emit_dist) {
    const JoinParams p = make_join_params(ix, out, emit_dist);
    TcParams t;
    t.rows_a = static_cast<const __nv_bfloat16*>(ix->rows_a);
    t.rows_b = static_cast<const __nv_bfloat16*>(ix->rows_b);
    t.nrows = ((ix->n + 7) & ~int64_t(7)) + kTcPadRows;
    t.error = reinterpret_cast<int*>(ix->counters + 4);
    t.ab_bf16 = ix->kernel == SJ_KERNEL_FILTER_FP16X2 ? 0u : 1u;
    switch (ix->kp) {
        case 16: return launch_k<16>(ix, p, t);
        case 32: return launch_k<32>(ix, p, t);
        case 64: return launch_k<64>(ix, p, t);
        case 112: return launch_k<112>(ix, p, t);
        case 208: return launch_k<208>(ix, p, t);
        case 400: return launch_k<400>(ix, p, t);
        default:
            set_error("no tensor-core kernel for K = %d", ix->kp);
            return SJ_ERR_UNSUPPORTED;
    }
}

}  // namespace sj
