// Per-query candidate scan (Algorithm 1 with one basis): for each query, the exact
// squared Euclidean distance (Eq. 1, fp32) to every point of every probed cone, the
// k nearest by (distance, id).  One warp to eight blocks of sixteen per query, rows
// straight from global memory.
//
// The staged scan (scan_plain.cu) streams a query's rows through shared memory, one
// bulk copy per cone; its producer, its per-row shuffles and its single-lane lists
// bounded it (cones of six rows: 22% of DRAM, 47% of the issue slots, 17 warps per
// SM).  Here nothing is staged: a lane looks up a probed cone, a warp scan lays 32
// cones' rows end to end, and eight row loads per lane are in flight at once.  Per
// batch of eight loads the distances are summed across lanes by halving -- a lane
// passes on half of its partial sums and keeps the other half, so a batch costs 7
// to 9 shuffles instead of 40, in the canonical order of additions
// (osann_device.cuh; only operands of an addition change sides).  The k best are a
// sorted list over the lanes, so an insertion is a ballot and a shift.  What bounds
// it now is the rows' reads (thin cones: 6.45 TB/s of DRAM, 0.96 of the copy rate).
// Measured (us, staged -> this): 10^4 queries, 128 cones of 5.9 rows of d = 128,
// k = 10, 2070 -> 556; 20000 queries, 64 cones of image patches, d = 64, k = 4, near
// matches excluded, 3400 -> 601; cones of 500 rows: d = 32, 10^4 queries, 16 cones,
// k = 10 4880 -> 841, k = 1 1563 -> 828; 20 queries, 20 cones 77 -> 27; d = 64, 300
// queries, 20 cones, k = 4 192 -> 132; d = 128, 3000 queries 4180 -> 2050.
#include <cooperative_groups.h>

#include "osann_device.cuh"
#include "osann_launch.h"

namespace osann {

namespace {

constexpr int U = 8;  // row loads in flight per lane
constexpr uint32_t NONE = 0xFFFFFFFFu;

struct QueryScanArgs {
    const float *xs, *Y;
    const uint32_t *offsets, *perm, *probes;
    const int64_t* query_src;
    int64_t Q, P_eff, grid_w;
    int d, d_pad, k, radius;
    const uint32_t* sel;  // LISTED: [count, q_0, ...]
    int team;     // warps that share the rows of 32 cones: a power of two that divides the query's warps
    int cluster;  // blocks per query
    uint32_t NC;
    int64_t* out_ids;
    float* out_d;
};
// (a parameter of its own: QueryScanArgs, grown by these, made the compiler keep fewer
// loads in flight in the forms that do not read them, 4 to 6% of their time)
struct QueryScanBig {
    uint32_t rows;    // rows of a cone that are too many for a warp (NONE: no cone is that large)
    uint32_t big;     // and for a team
    uint32_t* heavy;  // list [count, q_0, ...] of the queries left because of that
};

// TPR lanes per row, F float4 pieces each; W warps per block.  W = 1: a query per
// warp, four per block; otherwise a cluster of a.cluster blocks per query, in teams
// of a.team warps: a team takes 32 cones at a time, its warps those cones' rows by turns.
// LISTED: the clusters take the queries of a list made on the device by turns.
// BIG: a query that meets a cone of more than b.big rows (one may hold half the index)
// is not answered but put on a list, for a launch in which all its warps share it.
template <int TPR, int F, bool EXCL, int W, bool BIG, bool LISTED = false>
__global__ void __launch_bounds__(W == 1 ? 128 : 32 * W) query_scan_kernel(const QueryScanArgs a, const QueryScanBig b)
{
    constexpr int CPP = 32 / TPR;     // rows per load instruction
    constexpr int B = U * CPP;        // rows per batch: 8 .. 64
    constexpr int RL = B > 32 ? 2 : 1;  // batch rows looked up per lane
    constexpr int NV = TPR >= U ? 1 : U / TPR;  // row sums a lane ends with
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wb = W == 1 ? 0 : int(threadIdx.x >> 5);
    const int64_t count = LISTED ? int64_t(a.sel[0]) : a.Q;
    // (a long list of queries whose warps share every cone: a block each)
    const bool alone = LISTED && !BIG && a.team == W * a.cluster && count * 2 >= int64_t(gridDim.x);
    const unsigned blocks = W == 1 || alone ? 1u : unsigned(a.cluster), rank = W == 1 ? 0u : blockIdx.x % blocks;
    const int wq = int(rank) * W + wb;  // warp of the query
    const int64_t first =
        W == 1 ? int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5) : int64_t(blockIdx.x / blocks);
    for (int64_t at = first; at < count; at += LISTED ? int64_t(gridDim.x / blocks) : count) {
        const int64_t q = LISTED ? int64_t(a.sel[1 + at]) : at;
        const int g = lane / TPR, sub = lane % TPR;
        float4 qv[F];
        {
            const float* y = a.Y + q * int64_t(a.d);
#pragma unroll
            for (int f = 0; f < F; ++f) {
                const int c = 4 * (sub * F + f);
                qv[f].x = c + 0 < a.d ? y[c + 0] : 0.f;
                qv[f].y = c + 1 < a.d ? y[c + 1] : 0.f;
                qv[f].z = c + 2 < a.d ? y[c + 2] : 0.f;
                qv[f].w = c + 3 < a.d ? y[c + 3] : 0.f;
            }
        }
        const int64_t src = EXCL ? a.query_src[q] : -1;
        WarpTopk best;
        // the row index, inside its load group, whose sum this lane ends with (its
        // lowest for TPR < U), from the halving steps below: the top bit first
        int u0 = 0;
#pragma unroll
        for (int s = 0; (1 << s) < (TPR < U ? TPR : U); ++s) u0 |= ((lane >> s) & 1) << (2 - s);
        const bool primary = sub < U;  // (lanes that share a sum: one of them speaks)

        bool left = false;
        const uint32_t* pl = a.probes + q * a.P_eff;
        auto cone = [&](int64_t p, uint32_t& s0, uint32_t& n) {
            s0 = 0;
            n = 0;
            if (p < a.P_eff) {
                const uint32_t c = __ldg(pl + p);
                if (c < a.NC) {  // never produced by the probe kernel otherwise; guards the offsets read
                    s0 = __ldg(a.offsets + c);
                    n = __ldg(a.offsets + c + 1) - s0;
                    if (BIG && n > b.big) {
                        left = true;
                        n = 0;
                    }
                }
            }
        };
        const int team = W == 1 ? 1 : (alone ? W : a.team);
        const int64_t pbeg = W == 1 ? 0 : 32 * (wq / team), pstep = W == 1 ? 32 : 32 * (int(blocks) * W / team);
        const uint32_t tbeg = W == 1 ? 0u : uint32_t(wq % team * B), tstep = uint32_t(team * B);
        uint32_t st, sz;
        cone(pbeg + lane, st, sz);
        for (int64_t p0 = pbeg; p0 < a.P_eff; p0 += pstep) {
            uint32_t st1, sz1;
            cone(p0 + pstep + lane, st1, sz1);  // the next 32 cones, behind these ones' rows
            uint32_t incl = sz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            for (uint32_t t0 = tbeg; t0 < total; t0 += tstep) {
                // rows of the batch: lane l looks up rows l (and l + 32)
                uint32_t row[RL], id[RL];
#pragma unroll
                for (int h = 0; h < RL; ++h) {
                    const uint32_t t = t0 + uint32_t(32 * h + lane);
                    int c = 0;  // the first cone whose inclusive sum passes t
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1)
                        if (__shfl_sync(FULL, incl, c + w - 1) <= t) c += w;
                    const uint32_t r = __shfl_sync(FULL, st, c) + t -
                                       (__shfl_sync(FULL, incl, c) - __shfl_sync(FULL, sz, c));
                    const bool live = t < total && (B >= 32 || lane < B);
                    row[h] = live ? r : 0u;
                    id[h] = live ? __ldg(a.perm + r) : 0u;
                }
                float4 xv[U][F];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int e = u * CPP + g;
                    const uint32_t r = __shfl_sync(FULL, row[RL == 2 && u * CPP >= 32 ? RL - 1 : 0], e & 31);
                    const float4* xr = reinterpret_cast<const float4*>(a.xs + size_t(r) * a.d_pad) + sub * F;
#pragma unroll
                    for (int f = 0; f < F; ++f) xv[u][f] = __ldg(xr + f);
                }
                float v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float cp[F];
#pragma unroll
                    for (int f = 0; f < F; ++f) cp[f] = sq4(xv[u][f], qv[f]);
                    v[u] = pair_tree<F>(cp);
                }
                // pairwise tree across the TPR lanes: halving while a lane holds several sums
#pragma unroll
                for (int s = 0; (1 << s) < TPR; ++s) {
                    const int m = 1 << s;
                    const int half = U >> (s + 1);
                    if (half >= 1) {
                        const bool up = (lane >> s) & 1;
#pragma unroll
                        for (int i = 0; i < half; ++i) {
                            const float keep = up ? v[i + half] : v[i], give = up ? v[i] : v[i + half];
                            v[i] = keep + __shfl_xor_sync(FULL, give, m);
                        }
                    } else {
                        v[0] += __shfl_xor_sync(FULL, v[0], m);
                    }
                }
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const int e = (u0 + i) * CPP + g;
                    const uint32_t lo = __shfl_sync(FULL, id[0], e & 31);
                    const uint32_t hi = RL == 2 ? __shfl_sync(FULL, id[RL - 1], e & 31) : 0u;
                    const uint32_t cid = RL == 2 && e >= 32 ? hi : lo;
                    bool ok = primary && t0 + uint32_t(e) < total && v[i] <= di_dist(best.thr);
                    if (EXCL && ok && src >= 0) {
                        int64_t dr = int64_t(cid) / a.grid_w - src / a.grid_w;
                        int64_t dc = int64_t(cid) % a.grid_w - src % a.grid_w;
                        dr = dr < 0 ? -dr : dr;
                        dc = dc < 0 ? -dc : dc;
                        ok = (dr > dc ? dr : dc) > a.radius;
                    }
                    unsigned m = __ballot_sync(FULL, ok);
                    while (m) {
                        const int s = __ffs(int(m)) - 1;
                        m &= m - 1u;
                        best.insert(pack_di(__shfl_sync(FULL, v[i], s), __shfl_sync(FULL, cid, s)), a.k, lane);
                        m &= __ballot_sync(FULL, v[i] <= di_dist(best.thr));
                    }
                }
            }
            st = st1;
            sz = sz1;
        }
        if (BIG && W == 1) left = __any_sync(FULL, left);
        if (W > 1) {
            __shared__ uint64_t sh[W * 32];
            __shared__ int sh_left;
            if (lane < a.k) sh[wb * 32 + lane] = best.list;
            if (BIG) {
                left = __syncthreads_or(left);
                if (threadIdx.x == 0) sh_left = left;
            } else {
                __syncthreads();
            }
            if (W < 16) {
                if (wb == 0)
                    for (int w = 1; w < W; ++w)
                        for (int j = 0; j < a.k; ++j) best.insert(sh[w * 32 + j], a.k, lane);
            } else if (wb == 0) {
                // many lists: 32 entries at a time
                for (int i = a.k + lane; i - lane < W * a.k; i += 32)
                    best.offer(i < W * a.k, i < W * a.k ? sh[i / a.k * 32 + i % a.k] : EMPTY_DI, a.k, lane);
            }
            if (blocks > 1) {
                // the blocks' lists, through the first one's shared memory
                namespace cg = cooperative_groups;
                cg::cluster_group cl = cg::this_cluster();
                if (wb == 0 && lane < a.k) sh[lane] = best.list;
                cl.sync();
                if (rank == 0 && wb == 0)
                    for (unsigned r = 1; r < blocks; ++r) {
                        const uint64_t* rs = cl.map_shared_rank(sh, r);
                        best.offer(lane < a.k, lane < a.k ? rs[lane] : EMPTY_DI, a.k, lane);
                        if (BIG && *cl.map_shared_rank(&sh_left, r)) left = true;
                    }
                cl.sync();  // no block leaves, or goes on, while its list is read
            } else if (LISTED) {
                __syncthreads();
            }
        }
        if (BIG && left) {
            if (rank == 0 && wb == 0 && lane == 0) b.heavy[1 + atomicAdd(b.heavy, 1u)] = uint32_t(q);
        } else if (rank == 0 && wb == 0 && lane < a.k) {
            const uint32_t id = di_id(best.list);
            a.out_ids[q * a.k + lane] = id == 0xFFFFFFFFu ? int64_t(-1) : int64_t(id);
            a.out_d[q * a.k + lane] = di_dist(best.list);
        }
    }
}

// thin cones: a team per 32 probes, as far as the warps go; fat ones: all warps
int64_t team_of(int64_t P, int64_t warps, bool fat)
{
    int64_t team = warps;
    if (!fat)
        while (team > 1 && warps / team < (P + 31) / 32) team /= 2;
    return team;
}
// thin cones: waves of blocks (32 warps per SM) times a block's rounds of 32 probes
double rounds(int64_t Q, int64_t P, int64_t W, int num_sms)
{
    const int64_t slots = int64_t(num_sms) * 32 / W, team = team_of(P, W, false), teams = W / team;
    return double((Q + slots - 1) / slots) * double(((P + 31) / 32 + teams - 1) / teams) / double(team);
}

template <int TPR, int F, bool EXCL, int W, bool LISTED = false>
int launch_team(QueryScanArgs a, QueryScanBig b, bool fat, int cluster, int64_t clusters, cudaStream_t st)
{
    a.team = int(team_of(a.P_eff, int64_t(W) * cluster, fat));
    a.cluster = cluster;
    b.big = b.rows < NONE / uint32_t(a.team) ? b.rows * uint32_t(a.team) : NONE;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(clusters * cluster));
    cfg.blockDim = dim3(32 * W);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = unsigned(cluster);
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = b.rows != NONE ? cudaLaunchKernelEx(&cfg, query_scan_kernel<TPR, F, EXCL, W, true, LISTED>, a, b)
                                         : cudaLaunchKernelEx(&cfg, query_scan_kernel<TPR, F, EXCL, W, false, LISTED>, a, b);
    const int rc = count_launch();
    if (e != cudaSuccess && !rc) {
        set_error("per-query scan: launch failed (%s)", cudaGetErrorString(e));
        return -5;
    }
    return rc;
}

// Enough warps for the chip (some 3600 resident), and more, shorter blocks where a
// last wave of long ones would be nearly empty.  Measured (us):
//   thin cones, 1602 probes of 4.5 rows: W = 1 / 4 / 8 / 16 at 700 queries 934 / 383 /
//   394 / 310, 1268: 955 / 681 / 574 / 488, 2500: 1034 / 1026 / 942 / 846, 5000: 1332 /
//   1713 / 1678 / 1563; 128 probes of 6 rows, 700: 230 / 126 / 130 / 128, 1500: 242 /
//   197 / 179 / 190, 2500: 261 / 266 / 263 / 295;
//   patches (fat, uneven), 20 probes, 500: 184 / 91 / 75 / 75, 1000: 169 / 87 / 78 /
//   87, 3000: 227 / 124 / 129 / 171, 8000 (40 probes): 325 / 336 / 358 / 476.
// Over thin cones the number of warps whose blocks need the fewest rounds in all,
// which orders all of these but those bound by DRAM (795 queries, 260 probes: 165
// with sixteen warps, 141 with four; 550 probes: 348 with eight, 301 with four).  A tie goes to
// the shorter block, with many probes to the longer (900 queries, 1055 probes of 4.6 rows of
// d = 128: four warps 511, eight 554, sixteen 456; the staged scan 469).
// With sixteen, as many blocks, up to eight, as give every SM two (one / two / four /
// eight blocks: 24 queries, 198 cones of 17 rows of d = 100, 91 / 58 / 46 / 42; 6
// queries, 7000 thin cones, 210 / 132 / 97 / 72; 135 queries over patches 76 / 56 / 60
// / 93; 200 queries 48 / 56 / 60 / 83).  A list of queries takes eight: it is as often
// one query as all.
//
// Where a cone may be too large for a warp (b.rows), a launch of eight blocks per query
// follows for the queries with one (one, two, four, eight blocks: 4000 queries over thin
// cones of d = 64, some of them with a cone of 400 000 rows, 5744 / 2920 / 1509 / 803; left
// to their warps 35 600), except behind a form whose every query has sixteen warps on
// each cone.
template <int TPR, int F, bool EXCL>
int launch_listed(const QueryScanArgs& a, const QueryScanBig& b, bool fat, int num_sms, cudaStream_t st)
{
    const int64_t n = 2 * int64_t(num_sms) / 8, clusters = n < a.Q ? n : a.Q;
    return launch_team<TPR, F, EXCL, 16, true>(a, b, fat, 8, clusters < 1 ? 1 : clusters, st);
}
template <int TPR, int F, bool EXCL>
int launch_w(QueryScanArgs a, QueryScanBig b, bool fat, int num_sms, cudaStream_t st)
{
    int w = fat && a.Q >= 2048 ? 4 : (fat && a.Q >= 608 ? 8 : 16), c = 8;
    if (!fat && a.Q >= 256)
        for (const int v : {8, 4}) {
            const double r = rounds(a.Q, a.P_eff, v, num_sms), r0 = rounds(a.Q, a.P_eff, w, num_sms);
            if (r < r0 || (r == r0 && a.P_eff < 1024)) w = v;
        }
    if (a.Q >= (fat ? 6144 : (a.P_eff >= 256 ? 3600 : 2048))) w = 1;
    if (a.sel) w = 16;
    else if (w < 16) c = 1;
    while (!a.sel && c > 1 && a.Q * c > 2 * int64_t(num_sms)) c /= 2;
    if (team_of(a.P_eff, int64_t(w) * c, fat) >= 16) b.rows = NONE;
    const bool big = b.rows != NONE;
    if (big) cudaMemsetAsync(b.heavy, 0, 4, st);
    int rc;
    if (a.sel) {
        rc = launch_listed<TPR, F, EXCL>(a, b, fat, num_sms, st);
    } else if (w == 1) {
        b.big = b.rows;
        const unsigned blocks = unsigned((a.Q + 3) / 4);
        if (big) query_scan_kernel<TPR, F, EXCL, 1, true><<<blocks, 128, 0, st>>>(a, b);
        else query_scan_kernel<TPR, F, EXCL, 1, false><<<blocks, 128, 0, st>>>(a, b);
        rc = count_launch();
    } else {
        rc = w == 4 ? launch_team<TPR, F, EXCL, 4>(a, b, fat, 1, a.Q, st)
             : w == 8 ? launch_team<TPR, F, EXCL, 8>(a, b, fat, 1, a.Q, st)
                      : launch_team<TPR, F, EXCL, 16>(a, b, fat, c, a.Q, st);
    }
    if (rc || !big) return rc;
    a.sel = b.heavy;
    b.rows = NONE;
    return launch_listed<TPR, F, EXCL>(a, b, true, num_sms, st);
}

template <bool EXCL>
int launch_d(const QueryScanArgs& a, const QueryScanBig& b, bool fat, int num_sms, cudaStream_t st)
{
    switch (a.d_pad) {
    case 16: return launch_w<4, 1, EXCL>(a, b, fat, num_sms, st);
    case 32: return launch_w<8, 1, EXCL>(a, b, fat, num_sms, st);
    case 64: return launch_w<16, 1, EXCL>(a, b, fat, num_sms, st);
    case 128: return launch_w<32, 1, EXCL>(a, b, fat, num_sms, st);
    }
    return launch_w<32, 2, EXCL>(a, b, fat, num_sms, st);
}

}  // namespace

int launch_query_scan(const float* xs, const uint32_t* offsets, const uint32_t* perm, int d_pad, const float* Y, int d,
                     int64_t Q, const uint32_t* probes, int64_t P_eff, uint32_t NC, int k, const int64_t* query_src,
                     int64_t grid_w, int radius, bool fat, uint32_t warp_rows, uint32_t* scratch, const uint32_t* sel,
                     int num_sms, int64_t* out_ids, float* out_d, cudaStream_t st)
{
    if (Q == 0) return 0;
    QueryScanArgs a{};
    const QueryScanBig b{warp_rows, NONE, scratch};
    a.sel = sel;
    a.xs = xs;
    a.Y = Y;
    a.offsets = offsets;
    a.perm = perm;
    a.probes = probes;
    a.query_src = query_src;
    a.Q = Q;
    a.P_eff = P_eff;
    a.grid_w = grid_w;
    a.d = d;
    a.d_pad = d_pad;
    a.k = k;
    a.radius = radius;
    a.NC = NC;
    a.out_ids = out_ids;
    a.out_d = out_d;
    return query_src ? launch_d<true>(a, b, fat, num_sms, st) : launch_d<false>(a, b, fat, num_sms, st);
}

}  // namespace osann
