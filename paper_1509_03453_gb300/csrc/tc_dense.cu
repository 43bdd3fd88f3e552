// Dense screening: every row of the index against every query on the tensor
// cores, the survivors evaluated exactly.  Used for linear search (Eq. 1 over all
// N) and for searches whose cones are so thin that a tensor tile per cone would
// be padding (a 128-row tile for a cone of six rows), or whose survivor lists would
// overflow cone by cone (k > 1 and many candidates): there every row is screened and
// only survivors in a probed cone count.
//
// The screen (tc_scan_kernel.cuh) needs, per query, an upper bound U on its k-th
// best exact distance, and leaves about as many survivors as rows lie below it.
// So the rows are taken in phases, each seven times as many 128-row tiles as all
// the ones before it (tile numbers divisible by 8^n, then the rest divisible by
// 8^(n-1), ...; spread over the index, because neighbouring tiles hold neighbouring
// cones and a run of them can be all near one query): after a phase the survivors'
// exact distances are merged into the query's k best and U becomes the exact k-th, so
// that the next phase leaves about 8 k N / M survivors (M the candidates: all N rows in
// linear search), whatever N.  The seed of the first phase is exact too (query prep).  A query whose list overflows all the same (many rows within the error
// bound of each other), or that is out of the 16-bit range, is left to an exact
// scan of its own.
//
// What bounds it is the tensor core: 2 N Q d_pad (plus the 16 columns of the norm
// terms) fp16 operations, 0.3 ms for 1000 queries over 2*10^6 rows of d = 128;
// then the updates, whose chain survivor -> row -> list is latency.  Measured there
// with k = 10: 0.75 ms (0.95 with a register list per lane in seed and updates; the
// last phase's screen 0.26 ms); the fp32 tile scan 117.6 ms.
#include "osann.h"
#include "tc_scan_kernel.cuh"

namespace osann {

namespace {

constexpr int DENSE_U = 4;        // row passes with their loads in flight together
constexpr int DENSE_WARPS = 8;    // warps per block: of one query (small batches) or of as many queries
constexpr int DENSE_SMALL_Q = 4096;
constexpr int DENSE_SEED = 256;   // rows of the exact seed

__device__ __forceinline__ uint64_t cnk(const uint64_t* __restrict__ binom, int n, int k)
{
    if (n < 0 || k < 0 || k > n) return 0;
    return __ldg(binom + n * (MAX_L + 1) + k);
}

// Number of lexicographically smaller M-subsets of {0..n-1} than r[0] < ... < r[M-1].
template <int LM>
__device__ __forceinline__ uint64_t subset_rank(const uint64_t* __restrict__ binom, const int (&r)[LM], int first, int M,
                                                int base, int n)
{
    uint64_t rank = 0;
    int prev = 0;
#pragma unroll
    for (int j = 0; j < LM; ++j)
        if (j >= first && j < first + M) {
            // members prev .. v - 1 in this place: C(n - 1 - u, M - 1 - j) subsets each
            const int v = r[j] - base, left = M - (j - first);
            rank += cnk(binom, n - prev, left) - cnk(binom, n - v, left);
            prev = v + 1;
        }
    return rank;
}

// Position of cone `key` in a query's list (Sec. 3-B, probes.cu unranks the same
// order): inv[c] = the magnitude rank of component c, sg the query's sign words.
template <int L>
__device__ __forceinline__ uint64_t probe_position(uint32_t key, const uint8_t* inv, const uint32_t* sg, int d,
                                                   const uint64_t* __restrict__ binom)
{
    // members: the colex rank's largest members first
    uint64_t rest = key >> L;
    const uint32_t code = key & ((1u << L) - 1u);
    int rk[L];        // magnitude ranks, ascending
    uint32_t fl[L];   // differs from the query's sign
    int hi = d;
#pragma unroll
    for (int j = L - 1; j >= 0; --j) {
        int lo = j;   // largest s with C(s, j + 1) <= rest
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (cnk(binom, mid, j + 1) <= rest) lo = mid;
            else hi = mid;
        }
        rest -= cnk(binom, lo, j + 1);
        rk[j] = inv[lo];
        fl[j] = ((code >> (L - 1 - j)) ^ (sg[lo >> 5] >> (lo & 31))) & 1u;
        hi = lo;
    }
#pragma unroll
    for (int a = 1; a < L; ++a)
#pragma unroll
        for (int b = a; b > 0; --b)
            if (rk[b - 1] > rk[b]) {
                const int t = rk[b];
                rk[b] = rk[b - 1];
                rk[b - 1] = t;
                const uint32_t u = fl[b];
                fl[b] = fl[b - 1];
                fl[b - 1] = u;
            }
    // class: the members i_1..i_keep are kept
    int keep = 0, h = 0;
#pragma unroll
    for (int j = 0; j < L; ++j) {
        if (keep == j && rk[j] == j) ++keep;
        h += int(fl[j]);
    }
    const int delta = L - keep;
    uint64_t idx = delta > 0 ? 1 : 0;
#pragma unroll
    for (int t = 1; t < L; ++t)
        if (t < delta) idx += cnk(binom, d - L + t - 1, t);
    idx += subset_rank<L>(binom, rk, keep, delta, keep + 1, d - keep - 1);
    if (h == 0) return idx;
    // flipped cones: profile-major, subsets of the members by ascending magnitude
    const uint64_t nprof = cnk(binom, d, L);
    uint64_t before = 0;
#pragma unroll
    for (int t = 0; t < L; ++t)
        if (t < h) before += cnk(binom, L, t);
    int as[L];
    int n = 0;
#pragma unroll
    for (int t = 0; t < L; ++t) as[t] = 0;
#pragma unroll
    for (int t = 0; t < L; ++t)       // t: position by ascending magnitude
        if (fl[L - 1 - t]) {
#pragma unroll
            for (int u = 0; u < L; ++u)
                if (u == n) as[u] = t;
            ++n;
        }
    return nprof * before + idx * cnk(binom, L, h) + subset_rank<L>(binom, as, 0, h, 0, L);
}

struct UpdateArgs {
    const float *xs, *Y;
    int d, d_pad, k, cap, radius, first, last;
    int64_t Q, grid_w;
    const uint32_t* perm;
    const int64_t* query_src;
    uint32_t* surv_cnt;
    const uint32_t* surv;
    uint64_t* best;      // Q x k best so far
    uint32_t* Ubits;
    uint32_t* ovf;       // last phase: [count, q_0, ...]
    uint32_t* counter;   // work counter of the next phase
    unsigned long long* diag;
    int64_t* out_ids;
    float* out_d;
    DenseMember m;
};

// W warps per query, after each phase: the survivors that are candidates (not
// excluded; LC > 0: in a probed cone) merged into the query's k best by (canonical
// fp32 distance, id), the bound from the exact k-th; results after the last phase.
// LC: L of the member test, 0 for linear search.
template <int KMAX, int LC, int W>
__global__ void __launch_bounds__(32 * DENSE_WARPS) dense_update_kernel(const UpdateArgs a)
{
    constexpr int LM = LC > 0 ? LC : 1;
    __shared__ uint8_t inv_all[LC > 0 ? DENSE_WARPS : 1][MAX_D];
    __shared__ uint32_t row_all[DENSE_WARPS][32], id_all[DENSE_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wq = warp % W;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.counter = 0;
    const int64_t q = int64_t(blockIdx.x) * (DENSE_WARPS / W) + warp / W;
    if (q >= a.Q) return;  // W > 1: never
    const uint32_t n = a.surv_cnt[q];
    if (n > uint32_t(a.cap)) {
        // left to the exact scan: no further survivors are stored
        if (lane == 0 && wq == 0) {
            a.Ubits[q] = 0;
            if (a.last) {
                if (LC > 0) atomicAdd(a.diag + 1, 1ull);
                a.ovf[1 + atomicAdd(a.ovf, 1u)] = uint32_t(q);
            }
        }
        return;
    }
    const int n4 = a.d_pad >> 2;  // float4 pieces per row, one per lane (d_pad <= 128)
    const int CPP = 32 / n4;
    const int g = lane / n4, sub = lane % n4;
    float4 qv;
    {
        const float* y = a.Y + q * int64_t(a.d);
        const int c = 4 * sub;
        qv.x = c + 0 < a.d ? y[c + 0] : 0.f;
        qv.y = c + 1 < a.d ? y[c + 1] : 0.f;
        qv.z = c + 2 < a.d ? y[c + 2] : 0.f;
        qv.w = c + 3 < a.d ? y[c + 3] : 0.f;
    }
    const int64_t src = a.query_src ? a.query_src[q] : -1;
    uint8_t* inv = inv_all[LC > 0 ? warp : 0];
    uint32_t* rows = row_all[warp];
    uint32_t* ids = id_all[warp];
    if (LC > 0) {
        for (int r = lane; r < a.m.dk; r += 32) inv[a.m.qorder[q * a.m.dk + r]] = uint8_t(r);
        __syncwarp();
    }
    constexpr bool WARP_LIST = KMAX >= 16;  // k above 4: one list per warp, over its lanes
    WarpTopk wl;
    uint64_t list[KMAX];
    topk_init<KMAX>(list, a.k);
    if (WARP_LIST) {
        if (!a.first && wq == 0) wl.offer(lane < a.k, lane < a.k ? a.best[q * a.k + lane] : EMPTY_DI, a.k, lane);
    } else if (!a.first && wq == 0) {
        for (int j = lane; j < a.k; j += 32) {
            const uint64_t v = a.best[q * a.k + j];
            if (v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
        }
    }
    for (uint32_t b0 = uint32_t(32 * wq); b0 < n; b0 += 32 * W) {
        const bool live = b0 + lane < n;
        const uint32_t row = live ? a.surv[q * a.cap + b0 + lane] : 0u;
        const uint32_t id = live ? __ldg(a.perm + row) : 0u;
        bool ok = live;
        if (ok && src >= 0) {
            const int64_t dr = int64_t(id) / a.grid_w - src / a.grid_w, dc = int64_t(id) % a.grid_w - src % a.grid_w;
            const int64_t adr = dr < 0 ? -dr : dr, adc = dc < 0 ? -dc : dc;
            ok = (adr > adc ? adr : adc) > a.radius;
        }
        if (LC > 0 && ok)
            ok = probe_position<LM>(__ldg(a.m.keys + id), inv, a.m.qsign + q * (MAX_D / 32), a.m.dk, a.m.binom) <
                 uint64_t(a.m.P_eff);
        const unsigned mask = __ballot_sync(0xffffffffu, ok);
        if (ok) {
            const int at = __popc(mask & ((1u << lane) - 1u));
            rows[at] = row;
            ids[at] = id;
        }
        __syncwarp();
        const int m = __popc(mask);
        for (int i0 = 0; i0 < m; i0 += DENSE_U * CPP) {
            float4 xv[DENSE_U];
            int at[DENSE_U];
#pragma unroll
            for (int u = 0; u < DENSE_U; ++u) {
                at[u] = i0 + u * CPP + g;
                xv[u] = __ldg(reinterpret_cast<const float4*>(a.xs + size_t(rows[at[u] < m ? at[u] : 0]) * a.d_pad) + sub);
            }
#pragma unroll
            for (int u = 0; u < DENSE_U; ++u) {
                const float dist = lane_tree(sq4(xv[u], qv), n4);
                const bool is = sub == 0 && at[u] < m;
                const uint64_t v = pack_di(dist, is ? ids[at[u]] : 0u);
                if (WARP_LIST) wl.offer(is, v, a.k, lane);
                else if (is && v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
            }
        }
        __syncwarp();
    }
    if (W > 1) {
        // the warps' k best, gathered for the first one
        __shared__ uint64_t best_sh[W > 1 ? W * KMAX : 1];
        if (WARP_LIST) {
            if (lane < a.k) best_sh[wq * KMAX + lane] = wl.list;
        } else {
            for (int j = 0; j < a.k; ++j) {
                const uint64_t head = topk_head<KMAX>(list, a.k);
                const uint64_t b = warp_min_u64(head);
                if (head == b && b != EMPTY_DI) topk_remove<KMAX>(list, a.k, b);
                if (lane == 0) best_sh[wq * KMAX + j] = b;
            }
        }
        __syncthreads();
        if (wq != 0) return;
        topk_init<KMAX>(list, a.k);
        if (WARP_LIST) {
            for (int w = 1; w < W; ++w)
                wl.offer(lane < a.k, lane < a.k ? best_sh[w * KMAX + lane] : EMPTY_DI, a.k, lane);
        } else {
            for (int i = lane; i < W * a.k; i += 32) {
                const uint64_t v = best_sh[(i / a.k) * KMAX + i % a.k];
                if (v < list[KMAX - 1]) topk_insert<KMAX>(list, v);
            }
        }
    }
    if (LC > 0 && lane == 0) atomicAdd(a.diag, (unsigned long long)n);
    float kth = INFINITY;
    auto put = [&](int j, uint64_t b) {
        if (a.last) {
            const uint32_t id = di_id(b);
            a.out_ids[q * a.k + j] = id == 0xFFFFFFFFu ? int64_t(-1) : int64_t(id);
            a.out_d[q * a.k + j] = di_dist(b);
        } else {
            a.best[q * a.k + j] = b;
        }
    };
    if (WARP_LIST) {
        if (lane < a.k) put(lane, wl.list);
        kth = di_dist(wl.thr);
    } else {
        for (int j = 0; j < a.k; ++j) {
            const uint64_t head = topk_head<KMAX>(list, a.k);
            const uint64_t b = warp_min_u64(head);
            if (head == b && b != EMPTY_DI) topk_remove<KMAX>(list, a.k, b);
            kth = di_dist(b);
            if (lane == 0) put(j, b);
        }
    }
    if (lane == 0 && !a.last) {
        // the canonical fp32 distance is within 6.6e-7 relative of the exact one
        const float U = kth * (1.0f + 2e-6f) + 1e-30f;
        if (U < __uint_as_float(a.Ubits[q])) a.Ubits[q] = __float_as_uint(U);
        a.surv_cnt[q] = 0;
    }
}

size_t al(size_t x) { return (x + 255) / 256 * 256; }

struct Ws {
    size_t yb, qstat, ubits, scnt, surv, best, ovf, counter, total;
};
Ws ws_of(int64_t Q, int d_pad, int k)
{
    Ws w{};
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t o = off;
        off = al(off + b);
        return o;
    };
    w.yb = take(size_t(Q) * d_pad * 2);
    w.qstat = take(size_t(Q) * 16);
    w.ubits = take(size_t(Q) * 4);
    w.scnt = take(size_t(Q) * 4);
    w.surv = take(size_t(Q) * DENSE_SURV_CAP * 4);
    w.best = take(size_t(Q) * k * 8);
    w.ovf = take(size_t(Q + 1) * 4);
    w.counter = take(256);
    w.total = off;
    return w;
}

template <int LC, int W>
int launch_update_w(const UpdateArgs& u, cudaStream_t st)
{
    constexpr int per = DENSE_WARPS / W;
    const unsigned blocks = unsigned((u.Q + per - 1) / per);
    if (u.k <= 1) dense_update_kernel<1, LC, W><<<blocks, 32 * DENSE_WARPS, 0, st>>>(u);
    else if (u.k <= 4) dense_update_kernel<4, LC, W><<<blocks, 32 * DENSE_WARPS, 0, st>>>(u);
    else if (u.k <= 16) dense_update_kernel<16, LC, W><<<blocks, 32 * DENSE_WARPS, 0, st>>>(u);
    else dense_update_kernel<32, LC, W><<<blocks, 32 * DENSE_WARPS, 0, st>>>(u);
    return count_launch();
}

template <int LC>
int launch_update_k(const UpdateArgs& u, cudaStream_t st)
{
    return u.Q < DENSE_SMALL_Q ? launch_update_w<LC, DENSE_WARPS>(u, st) : launch_update_w<LC, 1>(u, st);
}

}  // namespace

int launch_tc_scan_dense(const void* maps, const TcArgs& a, bool debug, cudaStream_t st, int num_sms)
{
    return debug ? launch_tc_dense_dp<true>(maps, a, st, num_sms) : launch_tc_dense_dp<false>(maps, a, st, num_sms);
}

size_t dense_ws_bytes(int64_t Q, int d_pad, int k) { return ws_of(Q, d_pad, k).total; }
uint32_t* dense_ovf(void* ws, int64_t Q, int d_pad, int k)
{
    return reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + ws_of(Q, d_pad, k).ovf);
}

int launch_dense(const DenseIndex& ix, const float* Y, int64_t Q, int k, const int64_t* query_src, int64_t grid_w,
                 int radius, const DenseMember* member, void* ws, int64_t* out_ids, float* out_d, int debug,
                 cudaStream_t st, int num_sms)
{
    if (ix.d_pad > 128 || Q <= 0 || (member && (member->L < 1 || member->L > 4))) return -2;
    const Ws L = ws_of(Q, ix.d_pad, k);
    char* w = static_cast<char*>(ws);
    uint32_t* Ubits = reinterpret_cast<uint32_t*>(w + L.ubits);
    uint32_t* scnt = reinterpret_cast<uint32_t*>(w + L.scnt);
    uint32_t* surv = reinterpret_cast<uint32_t*>(w + L.surv);
    uint32_t* ovf = reinterpret_cast<uint32_t*>(w + L.ovf);
    uint32_t* counter = reinterpret_cast<uint32_t*>(w + L.counter);
    const int64_t seed = DENSE_SEED;
    int rc = launch_tc_query_prep(1, Y, Q, ix.d, ix.d_pad, member ? member->seed_probes : nullptr,
                                  member ? member->seed_P : 0, ix.N, ix.offsets, ix.NC, ix.xs, k, ix.cdot2, ix.cabs,
                                  ix.tcs, ix.perm, query_src, grid_w, radius, DENSE_SURV_CAP, w + L.yb,
                                  reinterpret_cast<float4*>(w + L.qstat), Ubits, scnt, st, int(seed), false);
    if (rc) return rc;
    cudaMemsetAsync(ovf, 0, 4, st);
    cudaMemsetAsync(counter, 0, 4, st);
    const int64_t groups = (Q + 2 * TC_GROUP - 1) / (2 * TC_GROUP);
    const int64_t T = (ix.N + TC_N - 1) / TC_N;
    int levels = 0;
    while ((ix.N >> (3 * levels)) > 16 * seed) ++levels;
    BatchedBuffers b{};
    b.counters = counter;
    UpdateArgs u{};
    u.xs = ix.xs;
    u.Y = Y;
    u.d = ix.d;
    u.d_pad = ix.d_pad;
    u.k = k;
    u.cap = DENSE_SURV_CAP;
    u.radius = radius;
    u.Q = Q;
    u.grid_w = grid_w;
    u.perm = ix.perm;
    u.query_src = query_src;
    u.surv_cnt = scnt;
    u.surv = surv;
    u.best = reinterpret_cast<uint64_t*>(w + L.best);
    u.Ubits = Ubits;
    u.ovf = ovf;
    u.counter = counter;
    u.diag = ix.diag;
    u.out_ids = out_ids;
    u.out_d = out_d;
    if (member) u.m = *member;
    for (int j = 0; j <= levels; ++j) {
        const int64_t mul = int64_t(1) << (3 * (levels - j));
        const int64_t all = (T + mul - 1) / mul;  // tiles divisible by mul
        TcDense dn{};
        dn.N = uint32_t(ix.N);
        dn.Q = uint32_t(Q);
        dn.tiles = uint32_t(j > 0 ? all - (all + 7) / 8 : all);
        dn.groups = uint32_t(groups);
        dn.mul = uint32_t(mul);
        dn.skip = j > 0 ? 1 : 0;
        // an item per SM at least, as far as the tiles go, and up to six of 32 tiles or
        // more: a new query tile costs about as much as three tiles
        int64_t chunks = (int64_t(num_sms) * 6 + groups - 1) / groups;
        if (chunks > dn.tiles / 32) chunks = dn.tiles / 32;
        const int64_t fill = (num_sms + groups - 1) / groups;
        if (chunks < fill) chunks = fill;
        if (chunks > dn.tiles) chunks = dn.tiles;
        dn.chunks = uint32_t(chunks);
        dn.n_items = uint32_t(chunks * groups);
        if (dn.n_items > 0) {
            rc = launch_tc_scan(1, ix.maps, ix.perm, ix.rowstat, w + L.yb, reinterpret_cast<float4*>(w + L.qstat), ix.tcs,
                                nullptr, 0, 0, b, Ubits, scnt, surv, DENSE_SURV_CAP, ix.status, ix.diag, ix.xs, Y, 1, ix.d,
                                ix.d_pad, 1, ix.cdot2, ix.Bn, ix.cabs, debug, st, num_sms,
                                int(seed), false, &dn);
            if (rc) return rc;
        }
        u.first = j == 0;
        u.last = j == levels;
        switch (member ? member->L : 0) {
        case 0: rc = launch_update_k<0>(u, st); break;
        case 1: rc = launch_update_k<1>(u, st); break;
        case 2: rc = launch_update_k<2>(u, st); break;
        case 3: rc = launch_update_k<3>(u, st); break;
        default: rc = launch_update_k<4>(u, st); break;
        }
        if (rc) return rc;
    }
    return 0;
}

}  // namespace osann
