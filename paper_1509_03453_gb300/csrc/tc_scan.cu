// Tensor-core screening path: query preparation (seed bounds, 16-bit query
// operands), the fp16 scale and row operands, tensor maps, the screening
// launch (kernel in tc_scan_kernel.cuh) and the exact fp32 rerank.
#include "osann.h"
#include "tc_scan_kernel.cuh"

namespace osann {

// ---------------------------------------------------------------- query prep

// 16-bit copy of -2 s y, scaled norms and A', survivor counter reset, and the
// initial upper bound U of each query: the k-th smallest canonical fp32 distance
// over a seed of rows (excluded rows skipped), inflated by the fp32 error bound;
// +inf if the seed holds fewer than k.  The seed is the rows of the first probed
// cones, in probe order, up to `seed_rows` (probes non-null), or `seed_rows` rows
// spread evenly over all N (probes null: linear search).  A query too large for
// the 16-bit range is left to an exact scan (its survivor count is set above the
// capacity), and so is every query when a row norm passed the fp32 range
// (tcs[3] = inf).
//
// The rows are read at random, so what bounds the kernel is the latency of the
// chain list entry -> cone offsets -> rows.  From prep_small_q queries up, a warp
// per query hides it behind the other warps and takes a cone at a time.  A small
// batch leaves the chip idle instead: there, PREP_SMALL warps share a query; 32
// probes are looked up at once (a lane each), the next 32 while these ones' rows
// are read, and a warp scan of the cone sizes lays thin cones end to end, so that
// every warp has TC_SEED_ILP row groups in flight.  Measured: 77 queries at
// d = 64, 132 -> 31 us; one query at d = 32, 49 -> 17 us; 4096 queries at d = 64,
// one warp each 28, the lookup of 32 cones 36 us.
constexpr int TC_SEED_ILP = 8;  // row groups loaded per iteration
constexpr int PREP_SMALL = 8;   // warps per query of a small batch
constexpr int PREP_WARP_LIST = 16;  // k above 4: one list per warp, over its lanes

// Rows scanned exactly for a query's initial bound.  A large batch keeps
// tightening its bounds as items finish, so a short seed suffices (64 rows
// from 4096 queries up; measured on 4096-query batches of d = 64 and 128,
// 64 rows halve this kernel's time and cost the screen and rerank less than
// that); in a small batch every item runs at once on the first bound, which
// must then be tighter (up to 1024 rows, a few cones): about 2^18 / Q rows,
// clamped.  For k > 4 the bound is the k-th best of the seed, and items of few
// rows hardly tighten it: k M / 64 rows, M the query's candidates, so that a few
// hundred of them stay below it, 64 to 1024 rows.  (1024 rows always, on
// two bases of 96 cones of 25 rows, k = 5, Q = 3001, took 650 us per basis beside
// a 280 us screen; on the thin-cone descriptor search, M = 72000, k = 10, 64 rows
// left 9.7 instead of 2.0 million survivors and overflowed lists.)
int tc_seed_rows(int64_t Q, int k, double M)
{
    const double r = k > 4 ? k * M / 64.0 : 0.0, q = Q > 0 ? (262144.0 + double(Q) - 1.0) / double(Q) : 1024.0;
    const double n = r > q ? r : q;
    return n < 64.0 ? 64 : (n > 1024.0 ? 1024 : int(n));
}

// Queries from which a warp each beats a block each.  The blocks shorten the chain, but
// keep the chip from the work list beside them: the sooner, the less a row's read takes
// and the more runs beside them (an index on a basis of its own, one of several searched at
// a time).  Whole searches with blocks / warps (us), k = 1: d = 16, 200 / 600 / 1000 queries
// 90 / 86, 97 / 89, 108 / 93; d = 50 on two bases, 871: 415 / 315; d = 64 on two, 552: 426 / 384;
// d = 128, fat cones on 16 PCA axes, 997: 432 / 374.  On the rows' own basis it is even from
// d = 32 up: d = 32, N = 10^6, 500 / 800: 132 / 122, 148 / 147; d = 50, N = 2.6*10^6, 756: 331 / 338,
// N = 3.5*10^5, 700: 190 / 206; d = 64, N = 4*10^6, 700: 366 / 318; d = 128, 500 / 1000: 304 / 384,
// 369 / 369.  k = 10, whose seed is longer: d = 16, 400 / 1000: 166 / 165, 198 / 171.
static int prep_small_q(int d_pad, int k, bool fat, bool rotated)
{
    if (d_pad <= 16) return k > 4 ? 512 : 128;
    if (!rotated) return 1024;
    if (d_pad <= 64 && k <= 4) return 512;
    return fat ? 900 : 1024;
}

struct PrepArgs {
    const float* Y;
    int64_t Q;
    int d, d_pad;
    const uint32_t* probes;  // null: the seed is spread over all N rows
    int64_t P_eff, N;
    const uint32_t* offsets;
    uint32_t NC;
    const float* xs;
    int k;
    float cdot2, cabs;
    const float* tcs;
    const uint32_t* perm;
    const int64_t* query_src;
    int64_t grid_w;
    int radius, cap, seed_rows;
    uint16_t* Y16;
    float4* qstat;
    uint32_t* Ubits;
    uint32_t* surv_cnt;
};

template <int F, int PREC, int KMAX>
__global__ void __launch_bounds__(128)
    tc_query_prep_kernel(const PrepArgs a)
{
    const float* const Y = a.Y;
    const int d = a.d, d_pad = a.d_pad, k = a.k, cap = a.cap, radius = a.radius, seed_rows = a.seed_rows;
    const int64_t Q = a.Q, P_eff = a.P_eff, grid_w = a.grid_w;
    const uint32_t* __restrict__ const probes = a.probes;
    const uint32_t* __restrict__ const offsets = a.offsets;
    const float* __restrict__ const xs = a.xs;
    const uint32_t NC = a.NC;
    const int lane = threadIdx.x & 31;
    const int64_t q = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    if (q >= Q) return;  // whole warp
    const float* y = Y + q * int64_t(d);
    const float sc = a.tcs[0];
    float s = 0.f, amax = 0.f;
    for (int c = lane * 4; c < d_pad; c += 128) {
        float4 v;
        v.x = c + 0 < d ? y[c + 0] : 0.f;
        v.y = c + 1 < d ? y[c + 1] : 0.f;
        v.z = c + 2 < d ? y[c + 2] : 0.f;
        v.w = c + 3 < d ? y[c + 3] : 0.f;
        // -2 s y: the factor is a power of two, so the 16-bit value is exact
        // up to the 16-bit rounding of s y itself
        uint2 pk;
        pk.x = pack16(to16_rn<PREC>(-2.f * sc * v.x), to16_rn<PREC>(-2.f * sc * v.y));
        pk.y = pack16(to16_rn<PREC>(-2.f * sc * v.z), to16_rn<PREC>(-2.f * sc * v.w));
        *reinterpret_cast<uint2*>(a.Y16 + q * int64_t(d_pad) + c) = pk;
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
        amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    }
    // fp16 holds |v| < 65504: keep 2 |s y| and the norm terms well inside (bf16: and the sums)
    const bool unscreenable = PREC == 1 ? 2.f * sc * amax > 16384.f || sc * sc * s > 32768.f : sc * sc * s > 1e30f;

    // seed rows: TPR lanes per row (canonical distance, as in the rerank)
    const int n4 = d_pad >> 2;
    const int TPR = n4 / F, CPP = 32 / TPR;
    const int g = lane / TPR, sub = lane % TPR;
    float4 qv[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
        const int c = 4 * (sub * F + f);
        qv[f].x = c + 0 < d ? y[c + 0] : 0.f;
        qv[f].y = c + 1 < d ? y[c + 1] : 0.f;
        qv[f].z = c + 2 < d ? y[c + 2] : 0.f;
        qv[f].w = c + 3 < d ? y[c + 3] : 0.f;
    }
    const int64_t src = a.query_src ? a.query_src[q] : -1;
    constexpr bool WARP_LIST = KMAX >= PREP_WARP_LIST;
    WarpTopk wl;
    uint64_t list[KMAX];
    topk_init<KMAX>(list, k);
    int scanned = 0;
    for (int64_t p = 0; p < P_eff && scanned < seed_rows; ++p) {
        const uint32_t b = probes[q * P_eff + p];
        if (b >= NC) continue;
        const uint32_t o0 = offsets[b], o1 = offsets[b + 1];
        for (uint32_t r0 = o0; r0 < o1 && scanned < seed_rows; r0 += TC_SEED_ILP * CPP) {
            // TC_SEED_ILP row groups per iteration: all loads in flight before the arithmetic
            float4 xv[TC_SEED_ILP][F];
            uint32_t rr[TC_SEED_ILP];
#pragma unroll
            for (int u = 0; u < TC_SEED_ILP; ++u) {
                rr[u] = r0 + uint32_t(u * CPP + g);
                const float4* xr =
                    reinterpret_cast<const float4*>(xs + size_t(rr[u] < o1 ? rr[u] : o0) * d_pad) + sub * F;
#pragma unroll
                for (int f = 0; f < F; ++f) xv[u][f] = xr[f];
            }
#pragma unroll
            for (int u = 0; u < TC_SEED_ILP; ++u) {
                float cpart[F];
#pragma unroll
                for (int f = 0; f < F; ++f) cpart[f] = sq4(xv[u][f], qv[f]);
                const float dist = lane_tree(pair_tree<F>(cpart), TPR);
                bool usable = rr[u] < o1;
                if (usable && src >= 0) {
                    // an excluded row is not a candidate and cannot seed the bound
                    const int64_t id = int64_t(a.perm[rr[u]]);
                    int64_t dr = id / grid_w - src / grid_w, dc = id % grid_w - src % grid_w;
                    dr = dr < 0 ? -dr : dr;
                    dc = dc < 0 ? -dc : dc;
                    usable = (dr > dc ? dr : dc) > radius;
                }
                const uint64_t v = pack_di(dist, rr[u]);
                if (WARP_LIST) wl.offer(sub == 0 && usable, v, k, lane);
                else if (sub == 0 && usable && v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
            }
            scanned += TC_SEED_ILP * CPP;
        }
    }
    // k-th smallest over the warp: k rounds of warp minimum over the lists
    float U = INFINITY;
    if (WARP_LIST) {
        // the canonical fp32 distance is within 6.6e-7 relative of the exact one
        if (wl.thr != EMPTY_DI) U = di_dist(wl.thr) * (1.0f + 2e-6f) + 1e-30f;
    } else {
        float kth = INFINITY;
        int found = 0;
        for (int j = 0; j < k; ++j) {
            const uint64_t head = topk_head<KMAX>(list, k);
            const uint64_t best = warp_min_u64(head);
            if (best == EMPTY_DI) break;
            if (head == best) topk_remove<KMAX>(list, k, best);
            kth = di_dist(best);
            ++found;
        }
        // the canonical fp32 distance is within 6.6e-7 relative of the exact one
        if (found == k) U = kth * (1.0f + 2e-6f) + 1e-30f;
    }
    if (lane == 0) {
        // scaled units: |q'| = s |q|; A' = 2c|q'| + Cabs, inflated by 2^-14
        // (16-bit hi/lo split of |x|) and rounded up to the 16-bit format
        const float qn = sc * sc * s, qnorm = sc * sqrtf(s);
        const float A = (a.cdot2 * qnorm + a.cabs) * (1.0f + 6.1035156e-5f);
        const float Ap = from16<PREC>(to16_ru<PREC>(A));
        a.qstat[q] = make_float4(qn, qnorm, -Ap, a.cabs * qnorm + tc_norm_eps(PREC));
        a.Ubits[q] = __float_as_uint(U);
        a.surv_cnt[q] = unscreenable || a.tcs[3] > 3.4e38f ? uint32_t(cap) + 1u : 0u;
    }
}

// The same for a small batch (a block per query), and for a seed spread over all
// rows (probes null).
template <int F, int PREC, int KMAX>
__global__ void __launch_bounds__(32 * PREP_SMALL) tc_query_prep_block_kernel(const PrepArgs a)
{
    constexpr int WPQ = PREP_SMALL;
    const int lane = threadIdx.x & 31, wq = int(threadIdx.x >> 5);  // warp of the query
    const int64_t q = blockIdx.x;
    const float* y = a.Y + q * int64_t(a.d);
    const float sc = a.tcs[0];

    // seed rows: TPR lanes per row (canonical distance, as in the rerank)
    const int n4 = a.d_pad >> 2;
    const int TPR = n4 / F, CPP = 32 / TPR;
    const int g = lane / TPR, sub = lane % TPR;
    float4 qv[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
        const int c = 4 * (sub * F + f);
        qv[f].x = c + 0 < a.d ? y[c + 0] : 0.f;
        qv[f].y = c + 1 < a.d ? y[c + 1] : 0.f;
        qv[f].z = c + 2 < a.d ? y[c + 2] : 0.f;
        qv[f].w = c + 3 < a.d ? y[c + 3] : 0.f;
    }
    const int64_t src = a.query_src ? a.query_src[q] : -1;
    constexpr bool WARP_LIST = KMAX >= PREP_WARP_LIST;
    WarpTopk wl;
    uint64_t list[KMAX];
    topk_init<KMAX>(list, a.k);
    // the rows t0 + u * CPP + g (u < TC_SEED_ILP) below `end`, row_of(t) -> row
    auto scan = [&](int t0, int end, auto row_of) {
        float4 xv[TC_SEED_ILP][F];
        uint32_t rr[TC_SEED_ILP];
        bool live[TC_SEED_ILP];
#pragma unroll
        for (int u = 0; u < TC_SEED_ILP; ++u) {
            const int t = t0 + u * CPP + g;
            live[u] = t < end;
            rr[u] = row_of(live[u] ? t : end - 1);
        }
#pragma unroll
        for (int u = 0; u < TC_SEED_ILP; ++u) {
            const float4* xr = reinterpret_cast<const float4*>(a.xs + size_t(rr[u]) * a.d_pad) + sub * F;
#pragma unroll
            for (int f = 0; f < F; ++f) xv[u][f] = xr[f];
        }
#pragma unroll
        for (int u = 0; u < TC_SEED_ILP; ++u) {
            float cpart[F];
#pragma unroll
            for (int f = 0; f < F; ++f) cpart[f] = sq4(xv[u][f], qv[f]);
            const float dist = lane_tree(pair_tree<F>(cpart), TPR);
            bool usable = live[u];
            if (usable && src >= 0) {
                // an excluded row is not a candidate and cannot seed the bound
                const int64_t id = int64_t(a.perm[rr[u]]);
                int64_t dr = id / a.grid_w - src / a.grid_w, dc = id % a.grid_w - src % a.grid_w;
                dr = dr < 0 ? -dr : dr;
                dc = dc < 0 ? -dc : dc;
                usable = (dr > dc ? dr : dc) > a.radius;
            }
            const uint64_t v = pack_di(dist, rr[u]);
            if (WARP_LIST) wl.offer(sub == 0 && usable, v, a.k, lane);
            else if (sub == 0 && usable && v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
        }
    };
    const int step = WPQ * TC_SEED_ILP * CPP;
    if (!a.probes) {
        for (int t0 = wq * TC_SEED_ILP * CPP; t0 < a.seed_rows; t0 += step)
            scan(t0, a.seed_rows, [&](int t) { return uint32_t(int64_t(t) * a.N / a.seed_rows); });
    } else {
        const uint32_t* pl = a.probes + q * a.P_eff;
        auto probe = [&](int64_t p) -> uint32_t { return p < a.P_eff ? pl[p] : 0xFFFFFFFFu; };
        uint32_t st = 0, sz = 0, b1 = probe(32 + lane);
        auto cone = [&](uint32_t b, uint32_t& s0, uint32_t& n) {
            s0 = 0;
            n = 0;
            if (b < a.NC) {
                s0 = a.offsets[b];
                n = a.offsets[b + 1] - s0;
            }
        };
        cone(probe(lane), st, sz);
        int scanned = 0;
        for (int64_t p0 = 0; p0 < a.P_eff && scanned < a.seed_rows; p0 += 32) {
            // the next 32 cones, and the probes after them
            uint32_t st1, sz1;
            cone(b1, st1, sz1);
            b1 = probe(p0 + 64 + lane);
            // no more rows of a cone than the seed still needs
            const uint32_t need = uint32_t(a.seed_rows - scanned);
            sz = sz < need ? sz : need;
            uint32_t incl = sz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
            const int total = int(all < need ? all : need);
            for (int t0 = wq * TC_SEED_ILP * CPP; t0 < total; t0 += step)
                scan(t0, total, [&](int t) {
                    // the first cone whose inclusive sum passes t
                    int c = 0;
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1)
                        if (__shfl_sync(0xffffffffu, incl, c + w - 1) <= uint32_t(t)) c += w;
                    return __shfl_sync(0xffffffffu, st, c) + uint32_t(t) -
                           (__shfl_sync(0xffffffffu, incl, c) - __shfl_sync(0xffffffffu, sz, c));
                });
            scanned += total;
            st = st1;
            sz = sz1;
        }
    }
    // k-th smallest: k rounds of warp minimum over each warp's lists, then over the
    // warps' k best, gathered in shared memory
    __shared__ uint64_t best_sh[WPQ * KMAX];
    float U = INFINITY;
    if (WARP_LIST) {
        best_sh[wq * KMAX + lane % KMAX] = EMPTY_DI;
        __syncwarp();
        if (lane < a.k) best_sh[wq * KMAX + lane] = wl.list;
        __syncthreads();
        if (wq != 0) return;
        for (int w = 1; w < WPQ; ++w)
            wl.offer(lane < a.k, best_sh[w * KMAX + lane % KMAX], a.k, lane);
        if (wl.thr != EMPTY_DI) U = di_dist(wl.thr) * (1.0f + 2e-6f) + 1e-30f;
    } else {
        float kth = INFINITY;
        int found = 0;
        auto rounds = [&](uint64_t* keep) {
            for (int j = 0; j < a.k; ++j) {
                const uint64_t head = topk_head<KMAX>(list, a.k);
                const uint64_t best = warp_min_u64(head);
                if (keep && lane == 0) keep[j] = best;
                if (best == EMPTY_DI) {
                    if (keep) continue;
                    break;
                }
                if (head == best) topk_remove<KMAX>(list, a.k, best);
                kth = di_dist(best);
                ++found;
            }
        };
        rounds(best_sh + wq * KMAX);
        __syncthreads();
        if (wq != 0) return;
        topk_init<KMAX>(list, a.k);
        for (int i = lane; i < WPQ * a.k; i += 32) {
            const uint64_t v = best_sh[(i / a.k) * KMAX + i % a.k];
            if (v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
        }
        found = 0;
        rounds(nullptr);
        // the canonical fp32 distance is within 6.6e-7 relative of the exact one
        if (found == a.k) U = kth * (1.0f + 2e-6f) + 1e-30f;
    }
    float s = 0.f, amax = 0.f;
    for (int c = lane * 4; c < a.d_pad; c += 128) {
        float4 v;
        v.x = c + 0 < a.d ? y[c + 0] : 0.f;
        v.y = c + 1 < a.d ? y[c + 1] : 0.f;
        v.z = c + 2 < a.d ? y[c + 2] : 0.f;
        v.w = c + 3 < a.d ? y[c + 3] : 0.f;
        // -2 s y: the factor is a power of two, so the 16-bit value is exact
        // up to the 16-bit rounding of s y itself
        uint2 pk;
        pk.x = pack16(to16_rn<PREC>(-2.f * sc * v.x), to16_rn<PREC>(-2.f * sc * v.y));
        pk.y = pack16(to16_rn<PREC>(-2.f * sc * v.z), to16_rn<PREC>(-2.f * sc * v.w));
        *reinterpret_cast<uint2*>(a.Y16 + q * int64_t(a.d_pad) + c) = pk;
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
        amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    }
    // fp16 holds |v| < 65504: keep 2 |s y| and the norm terms well inside (bf16: and the sums)
    const bool unscreenable = PREC == 1 ? 2.f * sc * amax > 16384.f || sc * sc * s > 32768.f : sc * sc * s > 1e30f;
    if (lane == 0) {
        // scaled units: |q'| = s |q|; A' = 2c|q'| + Cabs, inflated by 2^-14
        // (16-bit hi/lo split of |x|) and rounded up to the 16-bit format
        const float qn = sc * sc * s, qnorm = sc * sqrtf(s);
        const float A = (a.cdot2 * qnorm + a.cabs) * (1.0f + 6.1035156e-5f);
        const float Ap = from16<PREC>(to16_ru<PREC>(A));
        a.qstat[q] = make_float4(qn, qnorm, -Ap, a.cabs * qnorm + tc_norm_eps(PREC));
        a.Ubits[q] = __float_as_uint(U);
        a.surv_cnt[q] = unscreenable || a.tcs[3] > 3.4e38f ? uint32_t(a.cap) + 1u : 0u;
    }
}

// ---------------------------------------------------------------- rows

// The data scale of the screen: for fp16 the power of two with s^2 max|x|^2 <= 2^14
// (all-zero data: 1); for bf16 1, or that with <= 2^64 where the norms are larger (near
// fp32's limit the norm columns or the sums would overflow and lose rows).  tcs = (s, s^2, 1/s^2, X), X >= every row norm.
// The largest finite fp32 norm squared, below 2^128, needs s = 2^-57: s^2 and 1/s^2 are
// normal numbers, so nothing clamps the exponent from below (a scale too large would
// make the fp16 norm columns infinite and lose the row).  Above, s stays at 2^40:
// smaller norms only use less of the fp16 range.
template <int PREC>
__global__ void tc_scale_kernel(const uint32_t* __restrict__ maxn2_bits, float* __restrict__ tcs)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int e = 0;
    const float m = __uint_as_float(*maxn2_bits);  // +inf: a row's norm passed the fp32 range (nothing is screened)
    if (m > 0.0f && m < INFINITY) {
        int x;
        frexpf(m, &x);  // m < 2^x
        const int t = PREC == 1 ? 14 - x : (x > 64 ? 64 - x : 0);
        e = t >= 0 ? t / 2 : -((1 - t) / 2);
        e = e > 40 ? 40 : e;
    }
    const float sc = ldexpf(1.0f, e);
    tcs[0] = sc;
    tcs[1] = sc * sc;
    tcs[2] = 1.0f / (sc * sc);
    // a bound on every row norm, with room for the differently ordered fp32
    // sums of the per-row norms
    tcs[3] = sqrtf(m * (1.0f + 1e-4f)) * (1.0f + 1e-6f);
}

// 16-bit copy of s x (row-major, d_pad per row) and the extra K block of each
// row: 16-bit hi/lo splits of (1-B) s^2 |x|^2 and s |x|, then zeros.
template <int PREC>
__global__ void __launch_bounds__(256) tc_rows_kernel(const float* __restrict__ xs, const float4* __restrict__ rowstat,
                                                      int64_t N, int d_pad, const float* __restrict__ tcs,
                                                      uint16_t* __restrict__ x16, uint16_t* __restrict__ xe16)
{
    const float sc = tcs[0], sc2 = tcs[1];
    const int64_t n4 = N * (d_pad / 4);
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n4; i += int64_t(gridDim.x) * blockDim.x) {
        const float4 v = reinterpret_cast<const float4*>(xs)[i];
        uint2 pk;
        pk.x = pack16(to16_rn<PREC>(sc * v.x), to16_rn<PREC>(sc * v.y));
        pk.y = pack16(to16_rn<PREC>(sc * v.z), to16_rn<PREC>(sc * v.w));
        reinterpret_cast<uint2*>(x16)[i] = pk;
    }
    for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < N; r += int64_t(gridDim.x) * blockDim.x) {
        const float4 rs = rowstat[r];
        const float a = sc2 * rs.x, b = sc * rs.y;
        const uint16_t ah = to16_rn<PREC>(a), bh = to16_rn<PREC>(b);
        const uint16_t al = to16_rn<PREC>(a - from16<PREC>(ah)), bl = to16_rn<PREC>(b - from16<PREC>(bh));
        uint4* dst = reinterpret_cast<uint4*>(xe16 + r * 16);
        dst[0] = make_uint4(pack16(ah, al), pack16(bh, bl), 0u, 0u);
        dst[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

int launch_tc_scale(int prec, const uint32_t* maxn2_bits, float* tcs, cudaStream_t st)
{
    if (prec == 0) tc_scale_kernel<0><<<1, 32, 0, st>>>(maxn2_bits, tcs);
    else tc_scale_kernel<1><<<1, 32, 0, st>>>(maxn2_bits, tcs);
    return count_launch();
}

int launch_tc_rows(int prec, const float* xs, const float4* rowstat, int64_t N, int d_pad, const uint32_t* maxn2_bits,
                   float* tcs, void* x16, void* xe16, cudaStream_t st, int num_sms)
{
    if (prec == 0) tc_scale_kernel<0><<<1, 32, 0, st>>>(maxn2_bits, tcs);
    else tc_scale_kernel<1><<<1, 32, 0, st>>>(maxn2_bits, tcs);
    int rc = count_launch();
    if (rc || N == 0) return rc;
    int64_t blocks = (N * (d_pad / 4) + 255) / 256;
    if (blocks > int64_t(num_sms) * 16) blocks = int64_t(num_sms) * 16;
    if (prec == 0)
        tc_rows_kernel<0><<<unsigned(blocks), 256, 0, st>>>(xs, rowstat, N, d_pad, tcs, static_cast<uint16_t*>(x16),
                                                             static_cast<uint16_t*>(xe16));
    else
        tc_rows_kernel<1><<<unsigned(blocks), 256, 0, st>>>(xs, rowstat, N, d_pad, tcs, static_cast<uint16_t*>(x16),
                                                             static_cast<uint16_t*>(xe16));
    return count_launch();
}

// ---------------------------------------------------------------- rerank

constexpr int RR_U = 4;  // candidate passes with their loads in flight together

// One warp per query: canonical fp32 distance of every survivor (or, after
// an overflow, of every row of every probed cone), top-k by (distance, id).
template <int F, int KMAX, bool EXCL>
__global__ void __launch_bounds__(128) tc_rerank_kernel(const float* __restrict__ xs, int d_pad,
                                                        const uint32_t* __restrict__ perm,
                                                        const uint32_t* __restrict__ offsets, uint32_t NC,
                                                        const float* __restrict__ Y, int d, int64_t Q,
                                                        const uint32_t* __restrict__ probes, int64_t P_eff,
                                                        const uint32_t* __restrict__ surv_cnt,
                                                        const uint32_t* __restrict__ surv, int cap, int k,
                                                        const int64_t* __restrict__ query_src, int64_t grid_w,
                                                        int radius, unsigned long long* __restrict__ diag,
                                                        uint32_t* __restrict__ ovf, int64_t* __restrict__ out_ids,
                                                        float* __restrict__ out_d)
{
    const int lane = threadIdx.x & 31;
    const int64_t q = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    if (q >= Q) return;
    const int n4 = d_pad >> 2;
    const int TPR = n4 / F;         // lanes per candidate (<= 32)
    const int CPP = 32 / TPR;       // candidates per pass
    const int g = lane / TPR, sub = lane % TPR;
    float4 qv[F];
    {
        const float* y = Y + q * int64_t(d);
#pragma unroll
        for (int f = 0; f < F; ++f) {
            const int c = 4 * (sub * F + f);
            qv[f].x = c + 0 < d ? y[c + 0] : 0.f;
            qv[f].y = c + 1 < d ? y[c + 1] : 0.f;
            qv[f].z = c + 2 < d ? y[c + 2] : 0.f;
            qv[f].w = c + 3 < d ? y[c + 3] : 0.f;
        }
    }
    const int64_t src = EXCL ? query_src[q] : -1;
    constexpr bool WARP_LIST = KMAX >= PREP_WARP_LIST;
    WarpTopk wl;
    uint64_t list[KMAX];
    topk_init<KMAX>(list, k);
    // the candidate's canonical distance from its row chunk xv (this lane's F
    // float4 of the row)
    auto distance = [&](const float4 (&xv)[F]) {
        float cpart[F];
#pragma unroll
        for (int f = 0; f < F; ++f) cpart[f] = sq4(xv[f], qv[f]);
        return lane_tree(pair_tree<F>(cpart), TPR);
    };
    // the top-k update
    auto consider = [&](uint32_t id, bool valid, float dist) {
        bool ok = valid && sub == 0;
        if (EXCL && ok && src >= 0) {
            const int64_t dr = int64_t(id) / grid_w - src / grid_w;
            const int64_t dc = int64_t(id) % grid_w - src % grid_w;
            const int64_t adr = dr < 0 ? -dr : dr, adc = dc < 0 ? -dc : dc;
            ok = (adr > adc ? adr : adc) > radius;
        }
        const uint64_t v = pack_di(dist, id);
        if (WARP_LIST) wl.offer(ok, v, k, lane);
        else if (ok && v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
    };
    const uint32_t n = surv_cnt[q];
    if (n <= uint32_t(cap)) {
        // RR_U passes at a time: their survivor rows, then these rows and ids, are all
        // in flight before the first distance
        for (uint32_t b0 = 0; b0 < n; b0 += RR_U * uint32_t(CPP)) {
            uint32_t rows[RR_U];
            bool valid[RR_U];
#pragma unroll
            for (int u = 0; u < RR_U; ++u) {
                const uint32_t i = b0 + uint32_t(u * CPP + g);
                valid[u] = i < n;
                rows[u] = valid[u] ? surv[q * cap + i] : 0u;
            }
            float4 xv[RR_U][F];
            uint32_t ids[RR_U];
#pragma unroll
            for (int u = 0; u < RR_U; ++u) {
                const float4* xr = reinterpret_cast<const float4*>(xs + size_t(rows[u]) * d_pad) + sub * F;
#pragma unroll
                for (int f = 0; f < F; ++f) xv[u][f] = xr[f];
                ids[u] = __ldg(perm + rows[u]);
            }
            float dist[RR_U];
#pragma unroll
            for (int u = 0; u < RR_U; ++u) dist[u] = distance(xv[u]);
#pragma unroll
            for (int u = 0; u < RR_U; ++u) consider(ids[u], valid[u], dist[u]);
        }
        if (lane == 0) atomicAdd(diag, (unsigned long long)n);
    } else {
        // survivor list overflowed: the query is rescanned by the plain scan
        if (lane == 0) {
            atomicAdd(diag + 1, 1ull);
            ovf[1 + atomicAdd(ovf, 1u)] = uint32_t(q);
        }
        return;
    }
    if (WARP_LIST) {
        if (lane < k) {
            const uint32_t id = di_id(wl.list);
            out_ids[q * k + lane] = id == 0xFFFFFFFFu ? int64_t(-1) : int64_t(id);
            out_d[q * k + lane] = di_dist(wl.list);
        }
        return;
    }
    for (int j = 0; j < k; ++j) {
        const uint64_t head = topk_head<KMAX>(list, k);
        const uint64_t best = warp_min_u64(head);
        if (head == best && best != EMPTY_DI) topk_remove<KMAX>(list, k, best);
        if (lane == 0) {
            const uint32_t id = di_id(best);
            out_ids[q * k + j] = id == 0xFFFFFFFFu ? int64_t(-1) : int64_t(id);
            out_d[q * k + j] = di_dist(best);
        }
    }
}

// ---------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int tc_encode_rows_map(void* map_out, const void* x16, int64_t N, int d_pad, int prec)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult qr;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qr) !=
                cudaSuccess ||
            qr != cudaDriverEntryPointSuccess || !p) {
            cudaGetLastError();
            set_error("cuTensorMapEncodeTiled is not available");
            return -2;
        }
        fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    // d_pad == 0 encodes the 16-column extra block array instead
    const int width = d_pad > 0 ? d_pad : 16;
    const int row_bytes = d_pad > 0 ? tc_row_bytes(d_pad) : 32;
    const cuuint64_t dims[2] = {cuuint64_t(width), cuuint64_t(N)};
    const cuuint64_t strides[1] = {cuuint64_t(width) * 2};
    const cuuint32_t box[2] = {cuuint32_t(row_bytes / 2), cuuint32_t(TC_N)};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapSwizzle sw = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                                   : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                                      : CU_TENSOR_MAP_SWIZZLE_32B);
    CUresult r = fn(static_cast<CUtensorMap*>(map_out),
                    prec == 0 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                    const_cast<void*>(x16), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d)", int(r));
        return -5;
    }
    return 0;
}

size_t tc_map_bytes() { return 2 * sizeof(CUtensorMap); }

int launch_tc_query_prep(int prec, const float* Y, int64_t Q, int d, int d_pad, const uint32_t* probes,
                         int64_t P_eff, int64_t N, const uint32_t* offsets, uint32_t NC, const float* xs, int k,
                         float cdot2, float cabs, const float* tcs, const uint32_t* perm, const int64_t* query_src,
                         int64_t grid_w, int radius, int cap, void* Y16, float4* qstat, uint32_t* Ubits,
                         uint32_t* surv_cnt, cudaStream_t st, int seed_rows, bool rotated)
{
    if (Q == 0) return 0;
    PrepArgs a{};
    a.Y = Y;
    a.Q = Q;
    a.d = d;
    a.d_pad = d_pad;
    a.probes = probes;
    a.P_eff = P_eff;
    a.N = N;
    a.offsets = offsets;
    a.NC = NC;
    a.xs = xs;
    a.k = k;
    a.cdot2 = cdot2;
    a.cabs = cabs;
    a.tcs = tcs;
    a.perm = perm;
    a.query_src = query_src;
    a.grid_w = grid_w;
    a.radius = radius;
    a.cap = cap;
    a.seed_rows = seed_rows;
    a.Y16 = static_cast<uint16_t*>(Y16);
    a.qstat = qstat;
    a.Ubits = Ubits;
    a.surv_cnt = surv_cnt;
    // d_pad <= 128: one float4 piece per lane
    const bool small = Q < prep_small_q(d_pad, k, N >= 128 * int64_t(NC), rotated) || !probes;
#define OSANN_PREP(PR, KM)                                                                              \
    do {                                                                                                \
        if (small) tc_query_prep_block_kernel<1, PR, KM><<<unsigned(Q), 32 * PREP_SMALL, 0, st>>>(a);   \
        else tc_query_prep_kernel<1, PR, KM><<<unsigned((Q * 32 + 127) / 128), 128, 0, st>>>(a);        \
    } while (0)
#define OSANN_PREP_K(PR)             \
    if (k <= 1) OSANN_PREP(PR, 1);      \
    else if (k <= 4) OSANN_PREP(PR, 4); \
    else if (k <= 16) OSANN_PREP(PR, 16); \
    else OSANN_PREP(PR, 32);
    if (prec == 0) { OSANN_PREP_K(0) }
    else { OSANN_PREP_K(1) }
#undef OSANN_PREP_K
#undef OSANN_PREP
    return count_launch();
}

int launch_tc_scan(int prec, const void* maps, const uint32_t* perm, const float4* rowstat, const void* Y16,
                   const float4* qstat, const float* tcs, const int64_t* query_src, int64_t grid_w, int radius,
                   const BatchedBuffers& b, uint32_t* Ubits, uint32_t* surv_cnt, uint32_t* surv, int cap,
                   uint32_t* status, unsigned long long* diag, const float* xs, const float* Y, int64_t S, int d,
                   int d_pad, int k, float cdot2, float Bn, float cabs, int debug, cudaStream_t st, int num_sms,
                   int seed_rows, bool uneven, const TcDense* dense)
{
    TcArgs a{};
    // The k-th best of an item's rows beats the seed's only if the item holds k rows
    // below the seed's bound, of which it expects k rows / seed rows.  Keeping the k
    // bounds costs more than all else for k > 4, so items where that has a chance
    // below about 0.001 (Poisson: k c >= k, c = 0.25 at k = 5, 0.55 at k = 32) don't.
    // Measured: 6546 queries, k = 32, 182 cones of 95 rows of d = 96: screen 2750 -> 330 us.
    const double least = k > 4 ? (0.2 + 0.011 * k) * seed_rows : 0.0;
    a.tighten = uint32_t(least > k ? least : k);
    a.perm = perm;
    a.rowstat = rowstat;
    a.Y16 = static_cast<const uint16_t*>(Y16);
    a.qstat = qstat;
    a.tcs = tcs;
    a.query_src = query_src;
    a.items = b.items;
    if (dense) a.dense = *dense;
    a.n_items_dev = b.n_items_dev;
    a.qlist = b.qlist;
    a.counter = b.counters;
    a.Ubits = Ubits;
    a.surv_cnt = surv_cnt;
    a.surv = surv;
    a.status = status;
    a.diag = diag;
    a.xs = xs;
    a.Y = Y;
    a.S = S;
    a.grid_w = grid_w;
    a.d = d;
    a.d_pad = d_pad;
    a.k = k;
    a.radius = radius;
    a.cap = cap;
    a.prec = prec;
    a.ksteps = (d + 15) / 16;
    a.cdot2 = cdot2;
    a.Bn = Bn;
    a.cabs = cabs;
    const bool excl = query_src != nullptr;
    if (dense) return launch_tc_scan_dense(maps, a, debug != 0, st, num_sms);
    if (uneven && (excl || k > 1) && !debug) return launch_tc_scan_uneven(maps, a, k, excl, st, num_sms);
    if (excl) return launch_tc_scan_excl(maps, a, k, debug != 0, st, num_sms);
    if (debug) return launch_tc_scan_debug(maps, a, k, st, num_sms);
    return launch_tc_dp<false, false>(maps, a, k, st, num_sms);
}

int launch_tc_rerank(const float* xs, int d_pad, const uint32_t* perm, const uint32_t* offsets, uint32_t NC,
                     const float* Y, int d, int64_t Q, const uint32_t* probes, int64_t P_eff, const uint32_t* surv_cnt,
                     const uint32_t* surv, int cap, int k, const int64_t* query_src, int64_t grid_w, int radius,
                     unsigned long long* diag, uint32_t* ovf, int64_t* out_ids, float* out_d, cudaStream_t st)
{
    if (Q == 0) return 0;
    cudaMemsetAsync(ovf, 0, 4, st);
    const unsigned blocks = unsigned((Q * 32 + 127) / 128);
    const bool excl = query_src != nullptr;
#define OSANN_RR(F, KM)                                                                                           \
    do {                                                                                                          \
        if (excl)                                                                                                 \
            tc_rerank_kernel<F, KM, true><<<blocks, 128, 0, st>>>(xs, d_pad, perm, offsets, NC, Y, d, Q, probes,  \
                                                                  P_eff, surv_cnt, surv, cap, k, query_src,       \
                                                                  grid_w, radius, diag, ovf, out_ids, out_d);     \
        else                                                                                                      \
            tc_rerank_kernel<F, KM, false><<<blocks, 128, 0, st>>>(xs, d_pad, perm, offsets, NC, Y, d, Q, probes, \
                                                                   P_eff, surv_cnt, surv, cap, k, query_src,      \
                                                                   grid_w, radius, diag, ovf, out_ids, out_d);    \
    } while (0)
#define OSANN_RR_K(F)              \
    if (k <= 1) OSANN_RR(F, 1);    \
    else if (k <= 4) OSANN_RR(F, 4); \
    else if (k <= 16) OSANN_RR(F, 16); \
    else OSANN_RR(F, 32);
    if (d_pad <= 128) {
        OSANN_RR_K(1)
    } else {
        OSANN_RR_K(2)
    }
#undef OSANN_RR_K
#undef OSANN_RR
    return count_launch();
}

}  // namespace osann
