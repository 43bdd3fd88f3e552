// Tensor-core screening kernel: shared by the launchers of tc_scan.cu,
// tc_scan_excl.cu, tc_scan_uneven.cu, tc_dense.cu (checks off) and tc_scan_debug.cu (checks on).
//
// Batched candidate scan with 16-bit tensor-core screening and an exact fp32
// rerank.  The 16-bit operands are bf16 (unit roundoff u = 2^-8) or fp16
// (u = 2^-11, eight times tighter bound); for fp16 the data and queries are
// first multiplied by an exact power of two s, chosen from the largest row
// norm so that |s x|^2 <= 2^14, and all screening quantities are in those
// scaled units (distances scale by s^2, exactly).  Subnormal fp16 rounding
// adds an absolute error, covered by the terms Cabs(|x| + |q|) (the vectors) and eps
// (the norm columns).
//
// For a work item (cone c, group of up to 256 queries that probe it: two tiles) the
// squared distances are first estimated on the 5th-generation tensor cores
// as  d~ = |q|^2 + |x|^2 - 2 q~.x~  (q~, x~ rounded to bf16, products exact,
// fp32 accumulation in TMEM), M = 128 queries x N = 128 cone rows per MMA
// group and query tile, the cone rows streamed by TMA (2-D tensor map over the bf16 copy of
// the permuted vectors, swizzled K-major tiles).  Each query keeps an upper
// bound U on its k-th best exact distance; a row survives the screen when
//     d~ - E(q, x) <= U,   E = 2 c |q| |x| + B (|q|^2 + |x|^2) + Cabs (|x| + |q|) + eps,
// where c bounds the 16-bit rounding of both operands plus the fp32
// accumulation (c = 2u + u^2 + K 2^-20) and B the fp32 error of
// the norms, of their bf16 hi/lo split and a cushion for the fp32 rounding of
// the exact distance.  The per-row terms are folded into the product by one
// extra K block of 16 columns: the query side holds (1, 1, -A', -A') with
// A' >= 2c|q| rounded up to bf16, the row side (|x|^2 hi, lo, |x| hi, lo)
// with |x|^2 scaled by (1-B), so the accumulator is directly
//     D = (1-B)|x|^2 - A'|x| - 2 q.x     and a row survives iff
//     D <= U - (1-B)|q|^2.  A
// discarded row is therefore provably farther than some candidate already
// seen, so the survivors contain the exact top-k.  Survivors are appended to
// a per-query list; the rerank computes their canonical fp32 distance (the
// same expression as every other path) and selects the top-k, so the result
// is bit-identical to the fp32 paths.  A query whose list overflows is
// rescanned in full by the per-query scan (counted).
#pragma once

#include <cuda.h>

#include "osann_device.cuh"
#include "osann_launch.h"
#include "osann_tc.cuh"

namespace osann {

constexpr int TC_M = 128;  // queries per query tile = MMA M
constexpr int TC_N = 128;  // cone rows per tile = MMA N = TMEM columns

// 16-bit conversions: PREC 0 = bf16, 1 = fp16 (round to nearest or up)
template <int PREC>
__device__ __forceinline__ uint16_t to16_rn(float f)
{
    if (PREC == 0) return __bfloat16_as_ushort(__float2bfloat16_rn(f));
    return __half_as_ushort(__float2half_rn(f));
}
template <int PREC>
__device__ __forceinline__ uint16_t to16_ru(float f)
{
    if (PREC == 0) return __bfloat16_as_ushort(__float2bfloat16_ru(f));
    return __half_as_ushort(__float2half_ru(f));
}
template <int PREC>
__device__ __forceinline__ float from16(uint16_t h)
{
    if (PREC == 0) return __bfloat162float(__ushort_as_bfloat16(h));
    return __half2float(__ushort_as_half(h));
}
// the value 16-bit word of a number that the 16-bit type holds exactly, precision at run time
__device__ __forceinline__ uint16_t to16_exact(int prec, float f)
{
    return prec == 0 ? __bfloat16_as_ushort(__float2bfloat16_rn(f)) : __half_as_ushort(__float2half_rn(f));
}
// Absolute rounding error of a row's folded norm terms, scaled units: the low word of
// fp16(|x|^2) has a spacing of 2^-24 however small the norm, so the split is off by up
// to 2^-25 (twice that here); bf16 has fp32's exponent range.  It matters where the
// scale follows a far larger row: beside a row of norm 10^6, rows of norm 5 lost 1 in
// 60 of their queries' nearest neighbours without it.
__host__ __device__ constexpr float tc_norm_eps(int prec) { return prec == 0 ? 7.5e-37f : 5.9604645e-8f; }
__device__ __forceinline__ uint32_t pack16(uint16_t lo, uint16_t hi) { return uint32_t(lo) | (uint32_t(hi) << 16); }

__host__ __device__ constexpr int tc_row_bytes(int d_pad) { return d_pad >= 64 ? 128 : d_pad * 2; }

// Shared-memory plan of one CTA (one per SM): query-tile slots per query tile,
// cone-tile stages of TC_N rows, survivors buffered per screening thread.
// d_pad = 128 has room for one slot per query tile only (36 KB each): the two
// query tiles then reload in turn, each behind the other's MMAs.
constexpr int TC_SMEM_MAX = 232448 - 1024;  // 227 KB, less the alignment slack
constexpr int TC_QT = 2;                    // query tiles per item
__host__ __device__ constexpr int tc_tile_bytes(int dp) { return TC_M * dp * 2 + TC_M * 32; }
__host__ __device__ constexpr int tc_slots(int dp) { return dp >= 128 ? 1 : 2; }
constexpr int TC_SBUF = 4;                  // survivors buffered per screening thread
constexpr int TC_IQ = 4;                    // items in the queue
__host__ __device__ constexpr int tc_static_bytes(int dp)  // barriers, queue, constants, survivors: an upper bound
{
    return 1024 + TC_QT * tc_slots(dp) * (TC_M * 20 + 16) + TC_QT * TC_M * (TC_SBUF * 8 + TC_IQ * 4);
}
__host__ __device__ constexpr int tc_stages(int dp)
{
    const int s = (TC_SMEM_MAX - tc_static_bytes(dp) - TC_QT * tc_slots(dp) * tc_tile_bytes(dp)) / tc_tile_bytes(dp);
    return s > 8 ? 8 : s;
}

struct TcArgs {
    const uint32_t* perm;
    const float4* rowstat;    // per row: ((1-B)|x|^2, |x|, |x|^2, 0); N + TC_N rows
    const uint16_t* Y16;      // Q x d_pad, 16-bit -2 s y
    const float4* qstat;      // per query, scaled: (|q|^2, |q|, -A' (16-bit value, A' >= 2c|q| + Cabs), Cabs |q| + eps)
    const float* tcs;         // (s, s^2, 1/s^2, X): X bounds every row norm (unscaled)
    const int64_t* query_src;
    const uint4* items;       // (first row, end row, first slot, slot count)
    const uint32_t* n_items_dev;
    const uint32_t* qlist;    // list entries: query * S (+ position)
    TcDense dense;
    uint32_t* counter;
    uint32_t tighten;    // items of this many rows or more tighten the bounds
    uint32_t* Ubits;     // per query: upper bound on the k-th best distance (float bits)
    uint32_t* surv_cnt;  // per query
    uint32_t* surv;      // Q x cap rows
    uint32_t* status;
    unsigned long long* diag;  // [0] survivors, [1] fallbacks, [2] bound checks, [3] bound violations
    const float* xs;
    const float* Y;
    int64_t S;
    int64_t grid_w;
    int d, d_pad, k, radius, cap;
    int prec;     // 0 bf16, 1 fp16
    int ksteps;   // K steps of 16 columns that hold components: ceil(d / 16); the rest of d_pad is zero
    float cdot2;  // 2c
    float Bn;     // B
    float cabs;   // coefficient of the subnormal rounding terms
};

// Item descriptor passed from the producer to the loaders.
struct TcItem {
    uint32_t r0, r1;    // cone rows; r0 == 0xFFFFFFFF marks the end of the work
    uint32_t qbeg, qn;  // slot-list range of the query group
};
// What the issuer and the screening warps need of an item, passed with its query tile.
struct TcWork {
    uint32_t r0, nrows;  // nrows == 0 marks the end of the work
    uint32_t t0;         // number of the item's first cone tile (stage t0 mod S)
};
// First row of the t-th tile of chunk c of a dense phase.
__device__ __forceinline__ uint32_t dense_row(const TcDense& d, uint32_t c, uint32_t t)
{
    const uint32_t p = c + t * d.chunks;
    return (d.skip ? p + p / 7u + 1u : p) * d.mul * uint32_t(TC_N);
}
// An item's queries [off, off + 128) belong to query tile qt: both tiles of an
// item of more than 128 queries, else the tiles take the items in turn.
__device__ __forceinline__ bool tc_used(uint32_t qt, uint32_t it, uint32_t qn)
{
    return qn > uint32_t(TC_M) || (it & 1u) == qt;
}

// Warp roles (512 threads, one CTA per SM).  An item is a cone and up to 256
// queries, two query tiles of 128, so that every cone tile brought into shared
// memory is multiplied twice.  (One tile per item would need 74 to 82 bytes per
// cycle and SM from L2 at full tensor rate: TMA moved at most 72 in a streaming
// test, and that with 110 KB in flight.)
//   warp 0      fetches items and streams the cone tiles with TMA;
//   warps 1, 2  issue the MMAs of query tile 0 and 1, two accumulators of TC_N
//               columns each (all 512 TMEM columns);
//   warp 3      looks up the items' query indices (list entries) for the loaders;
//   warps 4-7   loaders, two per query tile: gather the queries' 16-bit rows by
//               16-byte asynchronous copies straight into the swizzled tile, and
//               the per-query constants;
//   warps 8-15  screening, four per query tile, a thread per query row = TMEM lane.
// Hand-offs are mbarriers: item queue (producer to loaders), cone tiles (full /
// empty, once per query tile), query tiles with their constants (full / empty),
// accumulators (full / empty).  Every wait is bounded; a timeout sets ST_TIMEOUT
// and makes all roles drop out.
//
// What bounds the kernel is the chain of hand-offs around each 128 x 128 tile
// (192 to 576 tensor-core cycles), so that chain is kept short:
//   - producer and issuers run as whole warps, with template widths, and elect one
//     lane for the TMA and MMA instructions only: with run-time widths and a
//     single-lane branch an MMA took 297 cycles to issue per CTA (64 of the
//     tensor core);
//   - one commit per tile.  A second one idles the tensor core for 70 to 80
//     cycles (streaming test, 5 MMAs per tile: 799 against 640 cycles per pair of
//     tiles), so the screening warps, woken by the commit, pass on that the cone
//     tile (and after the last one the query tile) is free;
//   - issuers and screening warps wait on no item queue: the loaders pass the item
//     on with its query tile;
//   - an accumulator is released when its values are in registers, before they
//     are looked at;
//   - the loaders find the items' query indices in shared memory, put there by
//     warp 3, so that one global latency and not two lies between a free query
//     slot and its new tile;
//   - survivors wait in shared memory across items and are appended a few at a
//     time: the atomic's round trip held a screening warp for some 1500 cycles
//     whenever an item left one (9% of a 4096-query batch at d = 64).
// Measured on 4096-query batches (us): d = 64 1050 -> 706, d = 128 1205 -> 988;
// d = 32, 10^4 queries 219 -> 166; before: one query tile per CTA, two CTAs per SM
// (d = 128: one, query tiles in tensor memory).
constexpr int TC_THREADS = 512;
constexpr int TC_STAGES_MAX = 8;
constexpr uint32_t TC_NACC = 2;  // accumulators of TC_N columns per query tile

// per-query constants of a query row, derived from (|q|^2, A', Cq, U)
struct TcQConst {
    float qn2;   // |q|^2 (scaled)
    float Uthr;  // s^2 U - (1-B)|q|^2 + Cq (scaled)
    float Aq1;   // A' (scaled)
    float U;     // upper bound on the k-th best exact distance (unscaled)
    float Cq;    // Cabs |q| + the norm terms' absolute error (scaled)
    float Uoff;  // (1+B)|q|^2 + 2B s^2 X^2 + 2A' s X + Cq, X >= every row norm (scaled)
};

// DEBUG: check every screened value against an fp32 evaluation of the
// folded product (a separate instantiation, so the check costs nothing when off)
// DENSE: the items of a.dense (k = 1 class, whatever the search's k: the bounds
// are left to the phases' exact updates).
// UNEVEN: a candidate's bound takes the row's own norm, a load, not the index's largest.
// (Norms over a factor of 100, k = 2, 7920 queries over cones of 86 rows of d = 64: 200 000
// survivors instead of 877 000, 463 -> 291 us; on even norms the loads cost 2 to 6%.)
template <int KMAX, bool EXCL, bool DEBUG, int DP, bool DENSE, bool UNEVEN>
__global__ void __launch_bounds__(TC_THREADS, 1)
    tc_scan_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap_x,
                   const TcArgs a)
{
    // k = 1 without exclusion: the minimum of a full chunk bounds the best
    // candidate directly, and survivors need only their row
    constexpr bool FAST = KMAX == 1 && !EXCL;
    // columns read at a time: with a long list of bounds 64 values would spill
    constexpr int CW = KMAX >= 16 ? 32 : 64;
    constexpr int row_bytes = tc_row_bytes(DP);
    constexpr int kblocks = DP >= 64 ? DP / 64 : 1;
    constexpr int epb = row_bytes / 2;
    constexpr int ksteps_pb = epb / 16;
    constexpr int mainT = TC_M * DP * 2;         // main part of a query or cone tile (TC_M = TC_N rows)
    constexpr int tileT = tc_tile_bytes(DP);     // with the extra K block: 16 elements per row
    constexpr int S = tc_stages(DP);
    constexpr uint32_t NA = uint32_t(tc_slots(DP)), NACC = TC_NACC;
    constexpr uint32_t TMEM_COLS = TC_QT * NACC * TC_N;
    static_assert(S >= 2 && S <= TC_STAGES_MAX, "cone-tile stages");

    extern __shared__ unsigned char smem_raw[];
    unsigned char* base =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* sA = base;                         // [TC_QT][NA] query tiles
    unsigned char* sB = base + TC_QT * NA * tileT;    // S cone tiles
    __shared__ __align__(8) uint64_t iq_full[TC_IQ], ix_full[TC_IQ], iq_empty[TC_IQ];
    __shared__ __align__(8) uint64_t bfull[TC_STAGES_MAX], bempty[TC_STAGES_MAX];
    __shared__ __align__(8) uint64_t afull_all[TC_QT][NA], aempty_all[TC_QT][NA];
    __shared__ __align__(8) uint64_t accfull_all[TC_QT][TC_NACC], accempty_all[TC_QT][TC_NACC];
    __shared__ TcItem iq[TC_IQ];
    __shared__ uint32_t iq_q[TC_IQ][TC_QT * TC_M];  // the items' query indices, 0xFFFFFFFF past the last
    __shared__ TcWork work_all[TC_QT][NA];
    __shared__ float4 qc_all[TC_QT][NA][TC_M];      // per query row (|q|^2, A', Cq, U)
    __shared__ uint32_t qidx_all[TC_QT][NA][TC_M];  // query index, 0xFFFFFFFF for an unused row
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    constexpr int SW = TC_QT * TC_M;
    // survivors buffered per screening thread: (row, query), with EXCL (row, value)
    __shared__ uint2 sbuf[TC_SBUF * SW];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t tx_bytes = uint32_t(tileT);
    const float sc = a.tcs[0], sc2 = a.tcs[1], inv_sc2 = a.tcs[2], xmax = a.tcs[3];

    if (warp == 1) {
        tmem_alloc(&tmem_base_sh, TMEM_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < TC_IQ; ++i) {
            mbar_init(&iq_full[i], 1);
            mbar_init(&ix_full[i], 1);
            mbar_init(&iq_empty[i], 4);  // loader warps
        }
        for (int s = 0; s < S; ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], TC_QT);  // once per query tile
        }
        for (int q = 0; q < TC_QT; ++q) {
            for (uint32_t b = 0; b < NA; ++b) {
                mbar_init(&afull_all[q][b], 64);  // the tile's loader threads
                mbar_init(&aempty_all[q][b], 4);  // one arrival per screening warp
            }
            for (uint32_t b = 0; b < NACC; ++b) {
                mbar_init(&accfull_all[q][b], 1);
                mbar_init(&accempty_all[q][b], 4);
            }
        }
        fence_mbar_init();
        abort_sh = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    // called by whole warps; the result is the same in every lane, so that the
    // warp stays converged for its collective instructions after a give-up
    auto give_up = [&](uint64_t* bar, uint32_t parity) -> bool {
        bool ok = false;
        if (!abort_sh) {
            ok = mbar_wait_bounded(bar, parity);
            if (!ok) {
                if (!abort_sh) atomicOr(a.status, ST_TIMEOUT);
                abort_sh = 1;
            }
        }
        return ok;
    };
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        bool ok = mbar_try_wait(bar, parity);
        if (!ok) ok = give_up(bar, parity);
        return __all_sync(0xffffffffu, ok);
    };

    // query tile of this warp's role, and its hand-offs
    const uint32_t qt = warp == 2 || warp == 6 || warp == 7 || warp >= 12 ? 1u : 0u;
    uint64_t* const afull = afull_all[qt];
    uint64_t* const aempty = aempty_all[qt];
    uint64_t* const accfull = accfull_all[qt];
    uint64_t* const accempty = accempty_all[qt];
    TcWork* const work = work_all[qt];

    if (warp == 0) {
        // ------------------------------------------------ producer (whole warp)
        const uint32_t n_items = DENSE ? a.dense.n_items : *a.n_items_dev;
        uint32_t it = 0, tc = 0, s = 0, s_ph = 0;
        // lane 0 fetches the next item's index and descriptor one publish ahead,
        // so their latency overlaps the current item's tiles
        uint4 pf = make_uint4(0xFFFFFFFFu, 0, 0, 0);
        auto fetch = [&]() {
            const uint32_t i = atomicAdd(a.counter, 1u);
            if (i >= n_items) {
                pf = make_uint4(0xFFFFFFFFu, 0, 0, 0);
            } else if (!DENSE) {
                pf = a.items[i];
            } else {
                // tile chunk (of this phase) and query group, the groups of a chunk in turn
                const uint32_t c = i / a.dense.groups, q0 = (i - c * a.dense.groups) * uint32_t(TC_QT * TC_M);
                const uint32_t n = a.dense.Q - q0;
                const uint32_t nt = (a.dense.tiles - c + a.dense.chunks - 1) / a.dense.chunks;
                pf = make_uint4(c, c + nt * TC_N, q0, n < uint32_t(TC_QT * TC_M) ? n : uint32_t(TC_QT * TC_M));
            }
        };
        if (lane == 0) fetch();
        auto publish = [&](uint32_t& r0, uint32_t& r1) -> bool {
            const uint32_t slot = it % TC_IQ;
            if (it >= TC_IQ && !wait(&iq_empty[slot], ((it / TC_IQ) - 1) & 1u)) return false;
            r0 = __shfl_sync(0xffffffffu, pf.x, 0);
            r1 = __shfl_sync(0xffffffffu, pf.y, 0);
            if (lane == 0) {
                iq[slot] = TcItem{pf.x, pf.y, pf.z, pf.w};
                mbar_arrive(&iq_full[slot]);
                if (r0 != 0xFFFFFFFFu) fetch();
            }
            ++it;
            return r0 != 0xFFFFFFFFu;
        };
        uint32_t cr0, cr1, nr0, nr1;
        bool have = publish(cr0, cr1), ok = true;
        while (have) {
            const bool have_next = publish(nr0, nr1);  // one item ahead of its tiles
            const int ntiles = int((cr1 - cr0 + TC_N - 1) / TC_N);
            for (int t = 0; t < ntiles; ++t, ++tc) {
                // stage s = tc mod S, s_ph = (tc / S) & 1: wait for the stage's previous use
                if (tc >= uint32_t(S) && !wait(&bempty[s], s_ph ^ 1u)) { ok = false; break; }
                const int y0 = DENSE ? int(dense_row(a.dense, cr0, uint32_t(t))) : int(cr0) + t * TC_N;
                unsigned char* dst = sB + s * uint32_t(tileT);
                if (elect_one()) {
                    mbar_arrive_expect_tx(&bfull[s], tx_bytes);
#pragma unroll
                    for (int kb = 0; kb < kblocks; ++kb)
                        tma_load_2d(dst + kb * TC_N * row_bytes, &tmap, kb * epb, y0, &bfull[s]);
                    tma_load_2d(dst + mainT, &tmap_x, 0, y0, &bfull[s]);
                }
                if (++s == uint32_t(S)) {
                    s = 0;
                    s_ph ^= 1u;
                }
            }
            if (!ok) break;
            cr0 = nr0;
            cr1 = nr1;
            have = have_next;
        }
        if (__any_sync(0xffffffffu, abort_sh != 0)) {
            // let the last tile issued into each stage land before shared memory goes away
            for (uint32_t g = tc > uint32_t(S) ? tc - uint32_t(S) : 0u; g < tc; ++g)
                mbar_wait_bounded(&bfull[g % uint32_t(S)], (g / uint32_t(S)) & 1u);
        }
    } else if (warp <= TC_QT) {
        // ------------------------------------------------ MMA issuer of query tile qt (whole warp)
        constexpr int KS = kblocks * ksteps_pb;  // <= 8
        const int ksteps = a.ksteps;             // those that hold components
        // instruction descriptor: a full tile, or its first 64 rows
        const uint32_t idesc = idesc_f16_f32(TC_M, TC_N, a.prec == 0 ? 1u : 0u);
        const uint32_t idesc_h = idesc_f16_f32(TC_M, TC_N / 2, a.prec == 0 ? 1u : 0u);
        // descriptors of this tile's slot 0 and of stage 0; a slot, a stage and a K step
        // add their byte offset / 16 to the 14-bit start-address field, which
        // never carries (shared memory is below 2^18 bytes)
        unsigned char* sA0 = sA + qt * NA * uint32_t(tileT);
        const uint64_t da0 = smem_desc_kmajor(smem_u32(sA0), row_bytes);
        const uint64_t db0 = smem_desc_kmajor(smem_u32(sB), row_bytes);
        const uint64_t dax0 = smem_desc_kmajor(smem_u32(sA0 + mainT), 32);
        const uint64_t dbx0 = smem_desc_kmajor(smem_u32(sB + mainT), 32);
        constexpr uint32_t step = uint32_t(tileT) >> 4;
        // Every issuer sees every cone tile, in order: one of an item that is not its
        // query tile's it only waits for and releases, so that no stage's phase
        // runs ahead of it.
        uint32_t tc = 0, ab = 0, ab_ph = 0, seen = 0, s = 0, s_ph = 0;
        for (;;) {
            if (!wait(&afull[ab], ab_ph)) break;
            const uint32_t nrows = __shfl_sync(0xffffffffu, work[ab].nrows, 0);
            const uint32_t t0 = __shfl_sync(0xffffffffu, work[ab].t0, 0);
            bool ok = true;
            for (; ok && seen < t0; ++seen) {
                ok = wait(&bfull[s], s_ph);
                if (ok && lane == 0) mbar_arrive(&bempty[s]);
                if (++s == uint32_t(S)) {
                    s = 0;
                    s_ph ^= 1u;
                }
            }
            if (!ok || nrows == 0) break;
            const int ntiles = int((nrows + TC_N - 1) / TC_N);
            seen += uint32_t(ntiles);
            const uint64_t da = da0 + ab * step, dax = dax0 + ab * step;
            for (int t = 0; t < ntiles; ++t, ++tc) {
                const uint32_t acc = tc % NACC, acc_ph = ((tc / NACC) - 1) & 1u;
                // the two waits together: their latencies overlap
                bool rb = mbar_try_wait(&bfull[s], s_ph);
                bool ra = tc < NACC || mbar_try_wait(&accempty[acc], acc_ph);
                if (!rb) rb = give_up(&bfull[s], s_ph);
                if (!ra) ra = give_up(&accempty[acc], acc_ph);
                if (!__all_sync(0xffffffffu, ra && rb)) { ok = false; break; }
                tc_fence_after();
                const uint64_t db = db0 + s * step, dbx = dbx0 + s * step;
                const uint32_t dt = tmem + (qt * NACC + acc) * TC_N;
                // the screening reads whole 64-column chunks: a last tile of at
                // most 64 rows needs only the first
                const uint32_t id = nrows - uint32_t(t) * TC_N <= TC_N / 2 ? idesc_h : idesc;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < KS; ++kk) {
                        const uint32_t ko = uint32_t((kk / ksteps_pb) * TC_M * row_bytes + (kk % ksteps_pb) * 32) >> 4;
                        if (kk < ksteps) mma_bf16_ss(dt, da + ko, db + ko, id, kk > 0 ? 1u : 0u);
                    }
                    // extra K block: |x|^2 and |x| terms folded into the product
                    mma_bf16_ss(dt, dax, dbx, id, 1u);
                    mma_commit(&accfull[acc]);
                }
                if (++s == uint32_t(S)) {
                    s = 0;
                    s_ph ^= 1u;
                }
            }
            if (!ok) break;
            if (++ab == NA) {
                ab = 0;
                ab_ph ^= 1u;
            }
        }
        if (abort_sh && tc > 0) mbar_wait_bounded(&accfull[(tc - 1) % NACC], ((tc - 1) / NACC) & 1u);
    } else if (warp == 3) {
        // ------------------------------------------------ query indices of the items
        const uint32_t dv = uint32_t(a.S);
        for (uint32_t it = 0;; ++it) {
            const uint32_t slot = it % TC_IQ;
            if (!wait(&iq_full[slot], (it / TC_IQ) & 1u)) break;
            const TcItem d = iq[slot];
            const bool end = d.r0 == 0xFFFFFFFFu;
            constexpr int E = TC_QT * TC_M / 32;
            uint32_t e[E];
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const uint32_t j = d.qbeg + uint32_t(lane + 32 * i);
                e[i] = !end && uint32_t(lane + 32 * i) < d.qn ? (DENSE ? j : a.qlist[j]) : 0u;
            }
#pragma unroll
            for (int i = 0; i < E; ++i)
                iq_q[slot][lane + 32 * i] =
                    !end && uint32_t(lane + 32 * i) < d.qn ? (dv == 1u ? e[i] : e[i] / dv) : 0xFFFFFFFFu;
            __syncwarp();
            if (lane == 0) mbar_arrive(&ix_full[slot]);
            if (end) break;
        }
    } else if (warp >= 4 && warp < 8) {
        // ------------------------------------------------ query tile loaders
        // per query tile, one warp gathers rows 0..63 and one rows 64..127; lane l
        // holds the indices and constants of rows rb + l and rb + 32 + l
        const int rb = 64 * (warp & 1);
        constexpr int cpr = DP / 8;          // 16-byte chunks per 16-bit query row (2, 4, 8 or 16)
        constexpr int cpb = row_bytes / 16;  // chunks per row of one K block of the tile
        uint32_t t0 = 0, nl = 0;
        for (uint32_t it = 0;; ++it) {
            const uint32_t slot = it % TC_IQ;
            if (!wait(&ix_full[slot], (it / TC_IQ) & 1u)) break;
            const TcItem d = iq[slot];
            // nrows = 0: the end mark
            const uint32_t nrows = d.r0 == 0xFFFFFFFFu ? 0u : d.r1 - d.r0;
            const bool mine = nrows == 0 || tc_used(qt, it, d.qn);
            const uint32_t off = (d.qn > uint32_t(TC_M) ? qt * TC_M : 0u) + rb + lane;
            const uint32_t qr[2] = {iq_q[slot][off], iq_q[slot][off + 32]};
            __syncwarp();
            if (lane == 0) mbar_arrive(&iq_empty[slot]);
            const uint32_t first = t0;
            t0 += (nrows + TC_N - 1) / TC_N;
            if (!mine) continue;
            const uint32_t ab = nl % NA;
            if (nl >= NA && !wait(&aempty[ab], ((nl / NA) - 1) & 1u)) break;
            ++nl;
            float4 qs[2];
            float Ur[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                qs[h] = make_float4(0.f, 0.f, 0.f, 0.f);
                Ur[h] = INFINITY;
                if (qr[h] != 0xFFFFFFFFu) {
                    qs[h] = a.qstat[qr[h]];
                    Ur[h] = __uint_as_float(__ldcg(a.Ubits + qr[h]));
                }
            }
            unsigned char* dstA = sA + (qt * NA + ab) * uint32_t(tileT);
            if (lane == 0 && rb == 0) work[ab] = TcWork{d.r0, nrows, first};
            if (nrows != 0) {
                // the warp's 64 16-bit rows as asynchronous 16-byte copies, every chunk
                // in flight at once, consecutive lanes on consecutive chunks of one row
                // (each instruction reads whole 32-byte sectors)
#pragma unroll
                for (int j = 0; j < 2 * cpr; ++j) {
                    const int i = lane + 32 * j;  // chunk of the warp's rows
                    const int rl = i / cpr, ch = i % cpr;
                    // rl < 32 for all lanes or for none: the source register is uniform
                    const uint32_t qs_src = __shfl_sync(0xffffffffu, j < cpr ? qr[0] : qr[1], rl & 31);
                    unsigned char* dst = dstA + (ch / cpb) * TC_M * row_bytes + swz_offset(rb + rl, ch % cpb, row_bytes);
                    if (qs_src != 0xFFFFFFFFu)
                        cp_async16(dst, reinterpret_cast<const uint4*>(a.Y16 + int64_t(qs_src) * DP) + ch);
                    else
                        *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = rb + lane + 32 * h;
                // extra block: (1, 1, -A', -A', 0, ...) against (|x|^2 hi, lo, |x| hi, lo, 0, ...)
                uint4 e0 = make_uint4(0, 0, 0, 0);
                if (qr[h] != 0xFFFFFFFFu) {
                    const uint16_t one = to16_exact(a.prec, 1.0f), na = to16_exact(a.prec, qs[h].z);
                    e0.x = pack16(one, one);
                    e0.y = pack16(na, na);
                }
                qc_all[qt][ab][r] = make_float4(qs[h].x, -qs[h].z, qs[h].w, Ur[h]);
                qidx_all[qt][ab][r] = qr[h];
                *reinterpret_cast<uint4*>(dstA + mainT + swz_offset(r, 0, 32)) = e0;
                *reinterpret_cast<uint4*>(dstA + mainT + swz_offset(r, 1, 32)) = make_uint4(0, 0, 0, 0);
            }
            // this thread's copies have landed; make them and the stores above
            // visible to the tensor core (async proxy)
            cp_async_wait_all();
            fence_proxy_async_smem();
            mbar_arrive(&afull[ab]);
            if (nrows == 0) break;
        }
        cp_async_wait_all();
    } else if (warp >= 8) {
        // ------------------------------------------------ screening of query tile qt
        const int er = 32 * (warp & 3) + lane;  // query row of the tile = TMEM lane
        const int sr = int(qt) * TC_M + er;     // this thread's column of the survivor buffer
        const uint32_t tl = tmem + (uint32_t(32 * (warp & 3)) << 16) + qt * NACC * TC_N;
        uint32_t tc = 0;
        int nb = 0;  // survivors buffered by this thread
        // append the buffered survivors to their queries' lists (the atomics in
        // flight together)
        auto flush = [&]() {
            uint2 e[TC_SBUF];
            uint32_t pos[TC_SBUF];
#pragma unroll
            for (int i = 0; i < TC_SBUF; ++i)
                if (i < nb) {
                    e[i] = sbuf[i * SW + sr];
                    pos[i] = atomicAdd(a.surv_cnt + e[i].y, 1u);
                }
#pragma unroll
            for (int i = 0; i < TC_SBUF; ++i)
                if (i < nb && pos[i] < uint32_t(a.cap)) a.surv[int64_t(e[i].y) * a.cap + pos[i]] = e[i].x;
            // overflowed: the exact scan has the query, later items keep nothing of it (k = 1
            // hardly overflows, and its launch lost 6 to 10% to this: 988 -> 1046 us)
            if constexpr (KMAX > 1) {
#pragma unroll
                for (int i = 0; i < TC_SBUF; ++i)
                    if (i < nb && pos[i] >= uint32_t(a.cap)) a.Ubits[e[i].y] = 0;
            }
            nb = 0;
        };
        for (uint32_t it = 0;; ++it) {
            const uint32_t ab = it % NA;
            if (!wait(&afull[ab], (it / NA) & 1u)) break;
            const TcWork wk = work[ab];
            if (wk.nrows == 0) break;
            const float4 q4 = qc_all[qt][ab][er];
            const uint32_t qi = qidx_all[qt][ab][er];
            const int ntiles = int((wk.nrows + TC_N - 1) / TC_N);
            uint32_t s = wk.t0 % uint32_t(S);
            TcQConst cur;
            cur.qn2 = q4.x;
            cur.Aq1 = q4.y;
            cur.Cq = q4.z;
            cur.U = q4.w;
            cur.Uthr = sc2 * q4.w - (1.0f - a.Bn) * q4.x + q4.z;
            cur.Uoff = (1.0f + a.Bn) * q4.x + 2.0f * a.Bn * (sc * xmax) * (sc * xmax) + 2.0f * q4.y * sc * xmax + q4.z;
            const float U0 = cur.U;
            const bool active = qi != 0xFFFFFFFFu;
            const int64_t q = active ? int64_t(qi) : 0;
            const int64_t src = EXCL && active ? a.query_src[q] : -1;
            float ubl[KMAX];  // k smallest upper bounds seen for this query in this item
#pragma unroll
            for (int u = 0; u < KMAX; ++u) ubl[u] = INFINITY;
            const bool tighten = wk.nrows >= a.tighten;
            // an upper bound on a candidate's distance from its accumulator value:
            // d~ + E <= D + Uoff (scaled units)
            auto bound_of = [&](float val, uint32_t row) {
                if constexpr (UNEVEN) {
                    const float sx = sc * __ldg(&a.rowstat[row].y);
                    const float off = (1.0f + a.Bn) * cur.qn2 + cur.Cq + 2.0f * sx * (a.Bn * sx + cur.Aq1);
                    return fmaxf((val + off) * (1.0f + 1e-6f) * inv_sc2, 0.0f);
                }
                return fmaxf((val + cur.Uoff) * (1.0f + 1e-6f) * inv_sc2, 0.0f);
            };
            auto bound = [&](float ub) {
                if (ub < cur.U) {
#pragma unroll
                    for (int u = KMAX - 1; u > 0; --u) {
                        const float pu = ubl[u - 1];
                        if (pu > ub) ubl[u] = pu;
                        else if (ubl[u] > ub) ubl[u] = ub;
                    }
                    if (ubl[0] > ub) ubl[0] = ub;
                }
                // the k-th smallest bound of k distinct candidates bounds the k-th best
                float kth = INFINITY;
#pragma unroll
                for (int u = 0; u < KMAX; ++u)
                    if (u == a.k - 1) kth = ubl[u];
                if (kth < cur.U) {
                    cur.U = kth;
                    cur.Uthr = sc2 * cur.U - (1.0f - a.Bn) * cur.qn2 + cur.Cq;
                }
            };
            // EXCL: append the buffered survivors, minus the excluded rows, to the
            // query's list, and tighten U with the others' upper bounds (deferred: a
            // stale U only admits more rows)
            auto flush_excl = [&]() {
                for (int i = 0; i < nb; ++i) {
                    const uint32_t row = sbuf[i * SW + sr].x;
                    const int64_t id = int64_t(__ldg(a.perm + row));
                    int64_t dr = id / a.grid_w - src / a.grid_w, dcc = id % a.grid_w - src % a.grid_w;
                    dr = dr < 0 ? -dr : dr;
                    dcc = dcc < 0 ? -dcc : dcc;
                    if (src >= 0 && (dr > dcc ? dr : dcc) <= a.radius) continue;
                    const uint32_t pos = atomicAdd(a.surv_cnt + q, 1u);
                    if (pos < uint32_t(a.cap)) a.surv[q * a.cap + pos] = row;
                    if (tighten) bound(bound_of(__uint_as_float(sbuf[i * SW + sr].y), row));
                }
                nb = 0;
            };
            bool ok = true;
            for (int t = 0; t < ntiles; ++t, ++tc) {
                const uint32_t acc = tc % NACC;
                if (!wait(&accfull[acc], (tc / NACC) & 1u)) { ok = false; break; }
                if (lane == 0) {
                    // the tile's MMAs have completed: its operands are free
                    if ((warp & 3) == 0) mbar_arrive(&bempty[s]);
                    if (t == ntiles - 1) mbar_arrive(&aempty[ab]);
                }
                if (++s == uint32_t(S)) s = 0;
                tc_fence_after();
                const int y0 = DENSE ? int(dense_row(a.dense, wk.r0, uint32_t(t))) : int(wk.r0) + t * TC_N;
                const int nvalid = min(TC_N, DENSE ? int(a.dense.N) - y0 : int(wk.nrows) - t * TC_N);
                for (int c0 = 0; c0 < nvalid; c0 += CW) {
                    float v[CW], m[CW / 32];
                    if constexpr (CW == 64) tmem_ld32x2_min(tl + uint32_t(acc * TC_N + c0), v, m[0], m[1]);
                    else tmem_ld32_min(tl + uint32_t(acc * TC_N + c0), v, m[0]);
                    if (c0 + CW >= nvalid) {
                        // the accumulator's values are in registers: one arrival per warp
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&accempty[acc]);
                    }
                    const float vmin = fminf(m[0], m[CW / 32 - 1]);
                    const int lim = nvalid - c0;
                    // columns past the item's rows (the next cone's, in the last
                    // tile) can only lower the minimum: the exact mask below drops them
                    if (active && vmin <= cur.Uthr) {
                        if (FAST && !DENSE && lim >= 64) {
                            // every column is a row of the item's cone, so the row at
                            // the minimum is a candidate within this bound
                            const float ub = fmaxf((vmin + cur.Uoff) * (1.0f + 1e-6f) * inv_sc2, 0.0f);
                            if (ub < cur.U) {
                                cur.U = ub;
                                cur.Uthr = sc2 * cur.U - (1.0f - a.Bn) * cur.qn2 + cur.Cq;
                            }
                        }
#pragma unroll
                        for (int h = 0; h < CW / 32; ++h) {
                            if (m[h] > cur.Uthr) continue;
                            uint32_t mask = 0;
#pragma unroll
                            for (int j = 0; j < 32; ++j) mask |= (v[32 * h + j] <= cur.Uthr ? 1u : 0u) << j;
                            // a masked column is +inf, which an unbounded U would admit
                            const int limh = lim - 32 * h;
                            if (limh < 32) mask &= limh <= 0 ? 0u : (1u << limh) - 1u;
                            while (mask) {
                                const int j = __ffs(int(mask)) - 1;
                                mask &= mask - 1u;
                                if (nb == TC_SBUF) {
                                    if (EXCL) flush_excl();
                                    else flush();
                                }
                                float val = 0.f;
                                if (!FAST) {
                                    val = v[32 * h];
#pragma unroll
                                    for (int u = 1; u < 32; ++u) val = u == j ? v[32 * h + u] : val;
                                }
                                if (!FAST && !EXCL && tighten) bound(bound_of(val, uint32_t(y0 + c0 + 32 * h + j)));
                                sbuf[nb * SW + sr] =
                                    make_uint2(uint32_t(y0 + c0 + 32 * h + j), EXCL ? __float_as_uint(val) : qi);
                                ++nb;
                            }
                        }
                    }
                    if (DEBUG && active) {
                        // folded product against an fp32 evaluation, one column per thread
                        const int col = CW == 64 ? lane + 32 * (c0 / 64 % 2) : lane;
                        if (col < lim) {
                            const int row = y0 + c0 + col;
                            const float* xr = a.xs + size_t(row) * DP;
                            const float* yr = a.Y + q * int64_t(a.d);
                            float dot = 0.f;
                            for (int i = 0; i < a.d; ++i) dot = fmaf(xr[i], yr[i], dot);
                            const float4 rs = __ldg(a.rowstat + row);
                            float mine = v[0];
#pragma unroll
                            for (int u = 1; u < CW; ++u) mine = u == col ? v[u] : mine;
                            const float ref = -2.0f * sc2 * dot + sc2 * rs.x - cur.Aq1 * sc * rs.y;
                            const float qnorm = sqrtf(cur.qn2);
                            const float lim2 = a.cdot2 * qnorm * sc * rs.y * 1.001f +
                                               4.0f * a.Bn * (cur.qn2 + sc2 * rs.z) +
                                               2.0f * a.cabs * (sc * rs.y + qnorm) + 2.0f * tc_norm_eps(a.prec) + 1e-30f;
                            atomicAdd(a.diag + 2, 1ull);
                            if (fabsf(mine - ref) > lim2) {
                                atomicAdd(a.diag + 3, 1ull);
                                atomicOr(a.status, ST_BOUND);
                            }
                        }
                    }
                }
            }
            if (!ok) break;
            if (EXCL) {
                flush_excl();
            } else if (__any_sync(0xffffffffu, nb > TC_SBUF / 2)) {
                flush();
            }
            if (active) {
                if (cur.U < U0) atomicMin(a.Ubits + q, __float_as_uint(fmaxf(cur.U, 0.0f)));
            }
        }
        if (!EXCL) flush();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

template <int KMAX, bool EXCL, bool DEBUG, int DP, bool DENSE = false, bool UNEVEN = false>
static int launch_tc_t(const void* maps, const TcArgs& a, cudaStream_t st, int num_sms)
{
    constexpr int need = 1024 + (TC_QT * tc_slots(DP) + tc_stages(DP)) * tc_tile_bytes(DP);
    // over half of an SM's shared memory: a CTA takes all of its TMEM columns
    constexpr int smem = need < 116 * 1024 ? 116 * 1024 : need;
    auto kern = tc_scan_kernel<KMAX, EXCL, DEBUG, DP, DENSE, UNEVEN>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaGetLastError();
    const CUtensorMap* m = static_cast<const CUtensorMap*>(maps);
    kern<<<unsigned(num_sms), TC_THREADS, smem, st>>>(m[0], m[1], a);
    return count_launch();
}

// Launch of one (exclusion, check, norms) class over k and the padded widths.
template <bool EXCL, bool DEBUG, bool UNEVEN, int DP>
static int launch_tc_k(const void* maps, const TcArgs& a, int k, cudaStream_t st, int num_sms)
{
    if constexpr (EXCL || !UNEVEN) {  // (k = 1 bounds by a chunk's minimum: no row of its own)
        if (k <= 1) return launch_tc_t<1, EXCL, DEBUG, DP, false, UNEVEN>(maps, a, st, num_sms);
    }
    if (k <= 4) return launch_tc_t<4, EXCL, DEBUG, DP, false, UNEVEN>(maps, a, st, num_sms);
    if (k <= 16) return launch_tc_t<16, EXCL, DEBUG, DP, false, UNEVEN>(maps, a, st, num_sms);
    return launch_tc_t<32, EXCL, DEBUG, DP, false, UNEVEN>(maps, a, st, num_sms);
}
template <bool EXCL, bool DEBUG, bool UNEVEN = false>
static int launch_tc_dp(const void* maps, const TcArgs& a, int k, cudaStream_t st, int num_sms)
{
    switch (a.d_pad) {
    case 16: return launch_tc_k<EXCL, DEBUG, UNEVEN, 16>(maps, a, k, st, num_sms);
    case 32: return launch_tc_k<EXCL, DEBUG, UNEVEN, 32>(maps, a, k, st, num_sms);
    case 64: return launch_tc_k<EXCL, DEBUG, UNEVEN, 64>(maps, a, k, st, num_sms);
    case 128: return launch_tc_k<EXCL, DEBUG, UNEVEN, 128>(maps, a, k, st, num_sms);
    }
    return -2;
}

// Launch of a dense phase.
template <bool DEBUG>
static int launch_tc_dense_dp(const void* maps, const TcArgs& a, cudaStream_t st, int num_sms)
{
    switch (a.d_pad) {
    case 16: return launch_tc_t<1, false, DEBUG, 16, true>(maps, a, st, num_sms);
    case 32: return launch_tc_t<1, false, DEBUG, 32, true>(maps, a, st, num_sms);
    case 64: return launch_tc_t<1, false, DEBUG, 64, true>(maps, a, st, num_sms);
    case 128: return launch_tc_t<1, false, DEBUG, 128, true>(maps, a, st, num_sms);
    }
    return -2;
}

// One translation unit per launch class (they compile in parallel):
// tc_scan_excl.cu: exclusion radius, bound check on or off
int launch_tc_scan_excl(const void* maps, const TcArgs& a, int k, bool debug, cudaStream_t st, int num_sms);
// tc_scan_uneven.cu: k > 1 or exclusion over rows of uneven norms
int launch_tc_scan_uneven(const void* maps, const TcArgs& a, int k, bool excl, cudaStream_t st, int num_sms);
// tc_dense.cu: a dense phase
int launch_tc_scan_dense(const void* maps, const TcArgs& a, bool debug, cudaStream_t st, int num_sms);
// tc_scan_debug.cu: the plain launch with the bound check compiled in
int launch_tc_scan_debug(const void* maps, const TcArgs& a, int k, cudaStream_t st, int num_sms);

}  // namespace osann
