// Queries answered one warp per query.  Two kinds arrive here:
//   - deferred: in the lane-per-query kernel their pruning key after seeding
//     was too large for a shared tile (e.g. a flight's first samples, whose
//     neighbours are far away); Algorithm 2 puts such unfinished lines
//     aside and carries on with the others -- they are finished here, where
//     the whole warp works on one query (32, 64 or 128 candidates by k);
//   - unsettled (window id stored as -1 - w): a point outside the tile's list
//     could belong to the first k, or a chain of distances that FP32 cannot
//     order was too long for the tile; here the pruning key is that of a later
//     rank (a deferred query that ends the same way is run again at once like
//     that).
//
// k_tnn_warp: the 32 lanes split the grid keys, the member segments and the
// member points of one query.  Its candidates are sorted 32-bit keys (the
// tile kernel's: the distance's upper bits above a slot), entry r * 32 + lane
// of the list in register r of a lane.  Up to 32 points at a time: the few
// that pass are inserted by ballot and shift, many are sorted across the warp
// and merged by a bitonic network of shuffles.  The next points are fetched
// while the present ones are merged.  Seeding visits cubes of keys of growing
// radius around the query's own key (cells in the plane, buckets backwards in
// time) until the list is full; inside a chunk of segments the nearest is
// always scanned first (Algorithm 2's nearest-first fetch).  The main phase
// is the exclusion criterion and stop rule of Algorithm 2 over the other
// keys.  To settle, the list's distances are taken again in FP32 and put in
// order, and chains of close keys are ranked by their FP64 distances, a lane
// per entry, however long a chain is.
// What bounds it is latency: one query is a chain of dependent L2 reads and
// merges.  64-bit lists in shared memory (sorted and merge-path merged per 32
// points), one key per lane and round and a queue ticket for every idle warp
// took 52 us for the 170 handed-over queries of 10,000 points, 72 us for the
// 4,400 of 400,000, 584 us for the 56,600 of 4,000,000 and 267 us for the
// 47,000 of a half-hour-lag nowcast; register lists 52 / 67 / 463 / 215, four
// keys per lane and round 32 / 49 / 355 / 199, the first entry per warp
// without a ticket 28 / 45 / 350 / 199.
// A query still unsettled goes to k_fallback_exact: the definition, with the
// FP64 distance taken only for the points that FP32 cannot rule out.
#pragma once
#include "tnn_device.cuh"
#include "tnn_grid.cuh"

#define WQ_MORE 28 // ranks beyond k that set the pruning key of an unsettled query
#define WQ_KEYS 4   // keys per lane and round
#define WQ_INSERT 4 // at most this many passing points are inserted one by one
#ifndef WQ_RSEED
#define WQ_RSEED 4 // largest radius of the seeding shells
#endif

typedef Slots<9> WqSlots; // a list holds at most 128 points

struct WarpSmem {
    union {
        int slot[WqSlots::n]; // point index of every slot
        struct {            // to settle:
            unsigned long long key[128]; // exact keys
            double d64[128];
        };
    };
    unsigned used[32]; // renumbering
    int pre[32];
    int kend[32 * WQ_KEYS]; // key ranges of the present round: ends and offsets
    int krel[32 * WQ_KEYS];
    unsigned long long count[4]; // bounds, distances, segments, FP64 distances
};

__host__ __device__ inline size_t fb_exact_smem_per_warp(int k_max)
{
    return (size_t)k_max * 32 * 12;
}

__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long v, int m)
{
    return __shfl_xor_sync(FULLMASK, v, m);
}

__device__ __forceinline__ int warp_incl_sum(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, v, o);
        if (lane >= o)
            v += t;
    }
    return v;
}

// Ascending order of one key per lane.
__device__ __forceinline__ unsigned wq_sort(unsigned v, int lane)
{
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const unsigned o = __shfl_xor_sync(FULLMASK, v, j);
            v = ((lane & k) == 0) == ((lane & j) == 0) ? min(v, o) : max(v, o);
        }
    return v;
}

// Merge a sorted key per lane into the list: the 32 NR smallest stay.
template <int NR> __device__ __forceinline__ void wq_merge(unsigned (&a)[NR], unsigned b, int lane)
{
    a[NR - 1] = min(a[NR - 1], __shfl_xor_sync(FULLMASK, b, 31));
#pragma unroll
    for (int h = NR / 2; h > 0; h >>= 1)
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if ((r & h) == 0)
                tg_cmpx(a[r], a[r + h]);
#pragma unroll
    for (int j = 16; j > 0; j >>= 1)
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const unsigned o = __shfl_xor_sync(FULLMASK, a[r], j);
            a[r] = (lane & j) == 0 ? min(a[r], o) : max(a[r], o);
        }
}

// Insert one key (the same in every lane).
template <int NR> __device__ __forceinline__ void wq_insert(unsigned (&a)[NR], unsigned key, int lane)
{
    int pos = 0;
#pragma unroll
    for (int r = 0; r < NR; ++r)
        pos += __popc(__ballot_sync(FULLMASK, a[r] < key));
#pragma unroll
    for (int r = NR - 1; r >= 0; --r) {
        unsigned prev = __shfl_up_sync(FULLMASK, a[r], 1);
        if (r > 0) {
            const unsigned last = __shfl_sync(FULLMASK, a[r > 0 ? r - 1 : 0], 31);
            prev = lane == 0 ? last : prev;
        }
        const int g = r * 32 + lane;
        a[r] = g < pos ? a[r] : g == pos ? key : prev;
    }
}

#ifndef TNN_WARP_MINB
#define TNN_WARP_MINB 6 // CTAs per SM (4 M points: 5 368 us, 6 350, 7 353; fewer spill less when few queries come)
#endif
// NR list registers per lane: 32 NR candidates, for k <= 32 NR - 16.  A single
// window (MANY false) is read from the kernel's parameters, so that its fields
// are constant operands and take no registers (handed-over queries of 4 M
// points 239 -> 221 us; the tile kernel gains nothing from it).
template <int NR, bool MANY>
__global__ void __launch_bounds__(TNN_WARPS_PER_CTA * 32, TNN_WARP_MINB)
    k_tnn_warp(const __grid_constant__ KnnLaunch L)
{
    __shared__ __align__(16) WarpSmem smem[TNN_WARPS_PER_CTA];
    const int lane = threadIdx.x & 31;
    WarpSmem &S = smem[threadIdx.x >> 5];
    pdl_trigger();
    pdl_wait();

    unsigned nfb = *(volatile unsigned *)&L.scr->n_fallback;
    if ((long long)nfb > L.fb_cap)
        nfb = (unsigned)L.fb_cap;
    if (lane < 4)
        S.count[lane] = 0;
    int2 ent = make_int2(0, 0);
    bool retry = false; // the same query again with the larger list
    float tau0 = INFINITY;
    // Dynamic queue (query costs differ by orders of magnitude) behind one
    // entry per warp, dealt out over the CTAs: thousands of warps asking the
    // counter at once, most of them in vain when few queries were handed
    // over, would wait on one another.
    unsigned e = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (bool first = true;; first = false) {
        if (!retry) {
            if (!first) {
                if (lane == 0)
                    e = atomicAdd(&L.scr->fb_next, 1u) + gridDim.x * TNN_WARPS_PER_CTA;
                e = __shfl_sync(FULLMASK, e, 0);
            }
            if (e >= nfb)
                break;
            ent = L.fb_list[e];
            tau0 = L.fb_tau[e];
        }
        const bool unsettled = retry || ent.x < 0;
        const int wid = ent.x < 0 ? -1 - ent.x : ent.x;
        unsigned n_lb = 0, n_pairs = 0, n_segs = 0, n_fp = 0; // this query's, of this lane
        const KnnWin *W = MANY ? L.wins + wid : &L.w0;
        const float4 q = W->q[ent.y];
        const QCtx c = make_qctx(W, q, true);
        const float s0 = W->sig[0], s1 = W->sig[1], s2 = W->sig[2], s3 = W->sig[3];
        const float4 *__restrict__ pts = W->pts;
        const GridDesc &G = W->grid;
        const int k = W->k;
        // rank whose key prunes: every point up to a little above it is seen
        const int C = unsettled ? min(k + WQ_MORE, 32 * NR - 1) : k;
        unsigned a[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            a[r] = TG_EMPTY;
        // A deferred query may arrive with a pruning key: at least k + 4
        // points lie at or below it.
        float tau = unsettled ? INFINITY : tau0;
        bool filled = false; // the list has its C-th key
        int base = 0;

        // one point per lane (j < 0: none), loaded as p
        auto consider = [&](int j, const float4 &p) {
            const float d = dist32(c, s0, s1, s2, s3, p);
            const bool in = j >= 0 && p.w < c.T32 && d <= tau;
            unsigned m = __ballot_sync(FULLMASK, in);
            n_pairs += j >= 0;
            if (!m)
                return;
            if (base > WqSlots::n - 32) {
                // renumber the slots the list still holds (at most 32 NR)
                __syncwarp();
                S.used[lane] = 0;
                __syncwarp();
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    if (a[r] != TG_EMPTY)
                        atomicOr(&S.used[(a[r] & WqSlots::mask) >> 5], 1u << (a[r] & 31u));
                __syncwarp();
                const unsigned u = S.used[lane];
                const int inc = warp_incl_sum(__popc(u), lane);
                S.pre[lane] = inc - __popc(u);
                base = __shfl_sync(FULLMASK, inc, 31);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const unsigned s = a[r] & WqSlots::mask;
                    if (a[r] != TG_EMPTY)
                        a[r] = (a[r] & ~WqSlots::mask) |
                               (unsigned)(S.pre[s >> 5] + __popc(S.used[s >> 5] & ((1u << (s & 31u)) - 1u)));
                }
#pragma unroll 1
                for (int w = 0; w < WqSlots::n / 32; ++w) {
                    const unsigned uw = S.used[w];
                    const int id = S.slot[w * 32 + lane];
                    __syncwarp();
                    if ((uw >> lane) & 1u)
                        S.slot[S.pre[w] + __popc(uw & ((1u << lane) - 1u))] = id;
                    __syncwarp();
                }
            }
            const int slot = base + __popc(m & ((1u << lane) - 1u));
            if (in)
                S.slot[slot] = j;
            base += __popc(m);
            const unsigned key = in ? WqSlots::key(d, (unsigned)slot) : TG_EMPTY;
            if (__popc(m) <= WQ_INSERT) {
#pragma unroll 1
                do {
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    wq_insert<NR>(a, __shfl_sync(FULLMASK, key, src), lane);
                } while (m);
            } else {
                wq_merge<NR>(a, wq_sort(key, lane), lane);
            }
            unsigned kc = a[0];
#pragma unroll
            for (int r = 1; r < NR; ++r)
                kc = (C - 1) >> 5 == r ? a[r] : kc;
            kc = __shfl_sync(FULLMASK, kc, (C - 1) & 31);
            filled = kc != TG_EMPTY;
            if (kc < TG_INF)
                tau = fminf(tau, fmaf(WqSlots::upper(kc), 0x1p-12f, WqSlots::upper(kc)) + 0x1p-98f);
        };
        // The member segments of every lane's keys ([klo, klo + kn) in key
        // order), 32 segments per step whatever key they belong to.
        auto visit_keys = [&](const int (&klo)[WQ_KEYS], const int (&kn)[WQ_KEYS]) {
            int sum = 0;
#pragma unroll
            for (int u = 0; u < WQ_KEYS; ++u)
                sum += kn[u];
            if (!__any_sync(FULLMASK, sum > 0))
                return;
            const int inc = warp_incl_sum(sum, lane);
            const int total = __shfl_sync(FULLMASK, inc, 31);
            __syncwarp();
            int at = inc - sum;
#pragma unroll
            for (int u = 0; u < WQ_KEYS; ++u) {
                S.krel[lane * WQ_KEYS + u] = klo[u] - at;
                at += kn[u];
                S.kend[lane * WQ_KEYS + u] = at;
            }
            __syncwarp();
#pragma unroll 1
            for (int b0 = 0; b0 < total; b0 += 32) {
                const int g = b0 + lane;
                unsigned score = TG_EMPTY; // bound above the lane
                int first = 0, cnt = 0;
                if (g < total) {
                    int lo = 0, hi = 32 * WQ_KEYS - 1; // smallest range with kend > g
#pragma unroll 1
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (S.kend[mid] > g)
                            hi = mid;
                        else
                            lo = mid + 1;
                    }
                    const float4 *src = G.gseg + 4 * (size_t)(S.krel[lo] + g);
                    const float4 r3 = __ldg(src + 3);
                    const float lb = seg_lb(c, s3, __ldg(src), __ldg(src + 1), __ldg(src + 2));
                    first = __float_as_int(r3.x);
                    cnt = __float_as_int(r3.y);
                    // truncated towards zero: still a lower bound
                    if (lb <= tau)
                        score = (__float_as_uint(lb) & ~31u) | (unsigned)lane;
                    n_lb++;
                }
                // up to 32 points of the nearest segments: this lane's index
                int lf = 0, lc = 0;
                auto gather = [&](int &j) -> bool {
                    int fill = 0;
                    j = -1;
#pragma unroll 1
                    while (fill < 32) {
                        if (lc == 0) {
                            const unsigned best = __reduce_min_sync(FULLMASK, score);
                            if (best == TG_EMPTY || !(__uint_as_float(best & ~31u) <= tau))
                                break;
                            const int w = best & 31u;
                            if (lane == w)
                                score = TG_EMPTY;
                            lf = __shfl_sync(FULLMASK, first, w);
                            lc = __shfl_sync(FULLMASK, cnt, w);
                            if (lane == 0) {
                                n_segs++;
                                if (L.dbg_seen)
                                    dbg_mark_seen(L, ent.y, lf, lc);
                            }
                        }
                        const int take = min(lc, 32 - fill);
                        if (lane >= fill && lane < fill + take)
                            j = lf + lane - fill;
                        lf += take;
                        lc -= take;
                        fill += take;
                    }
                    return fill > 0;
                };
                int j = -1;
                bool have = false;
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                do {
                    // the next points are on their way while these are merged
                    int jn;
                    const bool more = gather(jn);
                    float4 pn = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (jn >= 0)
                        pn = __ldg(pts + jn);
                    if (have)
                        consider(j, p);
                    j = jn;
                    p = pn;
                    have = more;
                } while (have);
            }
        };

        int bhi = -1;
        {
            const float fb = (c.T32 - G.t0) * G.inv_dt;
            if (fb >= 0.0f)
                bhi = (int)fminf(floorf(fb), (float)(G.nb - 1));
        }
        if (bhi >= 0) {
            const int hx = min(max((int)floorf((c.sx - G.x0) * G.inv_cell), 0), G.nx - 1);
            const int hy = min(max((int)floorf((c.sy - G.y0) * G.inv_cell), 0), G.ny - 1);
            const int rcover = max(max(max(hx, G.nx - 1 - hx), max(hy, G.ny - 1 - hy)), bhi);
            const float ext_max = __ldg(G.ext_max);
            // One loop hands visit_keys the keys of both phases, up to 128 per
            // round -- a round is a chain of dependent reads, so it takes as
            // many keys as four reads in flight per lane bring:
            // ---- seeding: cubes of growing radius around the query's key, the
            // first one whole, then shells up to radius WQ_RSEED (a query with
            // fewer than C valid points would otherwise grow the cube over the
            // whole grid; the main phase visits each causal bucket once
            // instead);
            // ---- main: buckets backwards, keys within reach, by bound, as
            // many buckets per round as fit.
            bool seeding = true;
            int rs = 0, nk = 0, t0 = 0;                // shell rs of side x side x (rs + 1) positions
            int b = bhi, cx0 = 0, cy0 = 0, wx = 1, nc = 1; // main: next bucket, the reach rectangle
            float inv_nc = 1.0f, inv_wx = 1.0f;        // positions per bucket (or age) and per row
#pragma unroll 1
            for (;;) {
                if (t0 >= nk) {
                    t0 = 0;
                    if (seeding && rs > 0 && (filled || rs >= rcover || rs >= WQ_RSEED)) {
                        seeding = false;
                        if (rs >= rcover)
                            break; // the shells covered every causal key
                    }
                    if (seeding) {
                        ++rs;
                        wx = 2 * rs + 1;
                        nc = wx * wx;
                        nk = nc * (rs + 1);
                        cx0 = hx - rs;
                        cy0 = hy - rs;
                        b = bhi;
                    } else {
                        // buckets the temporal bound still allows (a prefix)
                        const unsigned bm = __ballot_sync(
                            FULLMASK, b - lane >= 0 && time_lb(c, s3, __ldg(G.bpm + max(b - lane, 0))) <= tau);
                        const int nbk = bm == FULLMASK ? 32 : __ffs(~bm) - 1;
                        if (nbk == 0)
                            break;
                        const float R = sqrtf(tau) * (1.0f + 0x1p-18f) + ext_max + c.delta;
                        int cx1, cy1;
                        reach_cells(c.sx, c.sx, R, G.x0, G.inv_cell, G.nx, cx0, cx1);
                        reach_cells(c.sy, c.sy, R, G.y0, G.inv_cell, G.ny, cy0, cy1);
                        wx = cx1 - cx0 + 1;
                        nc = max(wx, 0) * max(cy1 - cy0 + 1, 0);
                        if (nc == 0)
                            break; // no cell within reach
                        nk = nc * max(1, min(nbk, 32 * WQ_KEYS / nc));
                    }
                    inv_nc = 1.0f / (float)nc;
                    inv_wx = 1.0f / (float)wx;
                }
                int klo[WQ_KEYS], kn[WQ_KEYS];
                int4 kr[WQ_KEYS];
                int kx[WQ_KEYS], ky[WQ_KEYS];
#pragma unroll
                for (int u = 0; u < WQ_KEYS; ++u) {
                    const int t = t0 + u * 32 + lane;
                    // quotients of integers below 2^21: exact
                    const int db = (int)(((float)t + 0.5f) * inv_nc), rem = t - db * nc;
                    const int dy = (int)(((float)rem + 0.5f) * inv_wx);
                    const int cx = cx0 + rem - dy * wx, cy = cy0 + dy, bk = b - db;
                    bool in = t < nk && bk >= 0 && cx >= 0 && cx < G.nx && cy >= 0 && cy < G.ny;
                    // what the seeding has visited (or, shell by shell, visits)
                    const int cheb = max(max(abs(cx - hx), abs(cy - hy)), bhi - bk);
                    in = in && (seeding ? (rs == 1 || cheb == rs) : cheb > rs);
                    kr[u] = in ? __ldg(G.krec + (bk * G.ncell + cy * G.nx + cx)) : make_int4(0, 0, 0, 0);
                    kx[u] = cx;
                    ky[u] = cy;
                }
#pragma unroll
                for (int u = 0; u < WQ_KEYS; ++u) {
                    klo[u] = kr[u].x;
                    kn[u] = kr[u].y - kr[u].x;
                    const float rx0 = G.x0 + (float)kx[u] * G.cell, ry0 = G.y0 + (float)ky[u] * G.cell;
                    if (!(cell_lb(c, s3, rx0, rx0 + G.cell, ry0, ry0 + G.cell, __int_as_float(kr[u].z),
                                  __int_as_float(kr[u].w)) <= tau))
                        kn[u] = 0;
                }
                t0 += 32 * WQ_KEYS;
                if (!seeding && t0 >= nk)
                    b -= nk / nc;
                visit_keys(klo, kn);
            }
        }
        // ---- settle
        __syncwarp();
        bool ok;
        {
            // Points outside the list lie at or above `bound` (none when the
            // pruning key never took effect and nothing left the list).
            float bound = tau;
            const unsigned last = __shfl_sync(FULLMASK, a[NR - 1], 31);
            if (last != TG_EMPTY)
                bound = fminf(bound, WqSlots::lower(last));
            int id[NR], n = 0;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                id[r] = a[r] != TG_EMPTY ? S.slot[a[r] & WqSlots::mask] : -1;
                n += __popc(__ballot_sync(FULLMASK, id[r] >= 0));
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                unsigned long long key = SENT;
                if (id[r] >= 0)
                    key = pack_key(dist32(c, s0, s1, s2, s3, __ldg(pts + id[r])), id[r]);
                S.key[r * 32 + lane] = key;
            }
            __syncwarp();
            // the truncated keys had them almost in order: odd-even exchanges
            bool swapped;
#pragma unroll 1
            do {
                swapped = false;
#pragma unroll 1
                for (int ph = 0; ph < 2; ++ph) {
                    for (int i = 2 * lane + ph; i + 1 < n; i += 64) {
                        const unsigned long long x = S.key[i], y = S.key[i + 1];
                        if (y < x) {
                            S.key[i] = y;
                            S.key[i + 1] = x;
                            swapped = true;
                        }
                    }
                    __syncwarp();
                }
            } while (__any_sync(FULLMASK, swapped));
            // entries certainly below every point outside; which are close to
            // their successor (or to the bound)
            int ne = 0;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int i = r * 32 + lane;
                ne += __popc(__ballot_sync(FULLMASK, i < n && !(key_d(S.key[i]) >= bound)));
            }
            const bool full = bound < INFINITY;
            unsigned cl[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int i = r * 32 + lane;
                bool close = false;
                if (i < ne) {
                    const float d = key_d(S.key[i]), lim = fmaf(d, 0x1p-17f, d) + 0x1p-100f;
                    close = i + 1 < ne ? key_d(S.key[i + 1]) <= lim : full && bound <= lim;
                }
                cl[r] = __ballot_sync(FULLMASK, close);
            }
            auto is_close = [&](int i) {
                unsigned w = cl[0];
#pragma unroll
                for (int r = 1; r < NR; ++r)
                    w = (i >> 5) == r ? cl[r] : w;
                return ((w >> (i & 31)) & 1u) != 0;
            };
            const bool exact_all = (W->flags & TNN_FLAG_EXACT_D2) != 0;
            // end of the chain that holds rank k
            int end = min(k, ne) - 1;
#pragma unroll 1
            while (end >= 0 && end < ne && is_close(end))
                ++end;
            // overflowed distances cannot be ranked here
            const bool over = n > 0 && !(key_d(S.key[n > 0 ? n - 1 : 0]) < INFINITY);
            ok = !over && !(full && ne < k) && end < ne;
            if (ok) {
                int32_t *oi = W->out_idx + (int64_t)ent.y * k;
                float *od = W->out_d2 + (int64_t)ent.y * k;
#pragma unroll 1
                for (int i = lane; i <= end; i += 32)
                    if (exact_all || is_close(i) || (i > 0 && is_close(i - 1))) {
                        S.d64[i] = dist64(W->sigd, q, __ldg(pts + key_i(S.key[i])));
                        n_fp++;
                    }
                __syncwarp();
#pragma unroll 1
                for (int i = lane; i < max(end + 1, k); i += 32) {
                    if (i > end) { // fewer than k valid points
                        oi[i] = -1;
                        od[i] = INFINITY;
                        continue;
                    }
                    const unsigned long long key = S.key[i];
                    const bool chain = is_close(i) || (i > 0 && is_close(i - 1));
                    int rank = i;
                    if (chain) {
                        int t = i;
                        while (t > 0 && is_close(t - 1))
                            --t;
                        rank = t;
                        const double d = S.d64[i];
                        for (;; ++t) {
                            const double o = S.d64[t];
                            rank += o < d || (o == d && key_i(S.key[t]) < key_i(key));
                            if (!is_close(t))
                                break;
                        }
                    }
                    if (rank < k) {
                        oi[rank] = key_i(key);
                        od[rank] = chain || exact_all ? (float)S.d64[i] : key_d(key);
                    }
                }
            }
        }
        // a chain ran past the pruning key of rank k: once more with that of a
        // later rank before the FP64 definition is used
        retry = !ok && !unsettled;
        if (!ok && !retry && lane == 0) {
            const unsigned slot = atomicAdd(&L.scr->n_fallback3, 1u);
            if (slot < (unsigned long long)L.fb_cap)
                L.fb_list3[slot] = make_int2(wid, ent.y);
            else
                atomicOr(&L.scr->status, 2u);
        }
        const unsigned v[4] = {n_lb, n_pairs, n_segs, n_fp};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned x = __reduce_add_sync(FULLMASK, v[i]); // at most the index's points
            if (lane == 0)
                S.count[i] += x;
        }
        __syncwarp();
    }
    __syncwarp();
    if (lane < 4 && S.count[lane])
        atomicAdd(&L.scr->stats[1 + lane], S.count[lane]);
    if (blockIdx.x == 0 && threadIdx.x == 0)
        L.scr->stats[5] = nfb;
}

// Fault flags of the search launches on this device (the bits of
// KnnScratch::status: 1 and 2 a fallback list overflowed, 4 a bounded wait
// timed out), ORed in by the last kernel of every search and kept until a
// synchronising call reports and clears them (tnn_sync_status).  Searches
// without statistics and tnn_knn_noalloc report through it.
static __device__ unsigned int g_search_fault;

__global__ void __launch_bounds__(TNN_WARPS_PER_CTA * 32)
    k_fallback_exact(const __grid_constant__ KnnLaunch L)
{
    // After the wait the kernels before this one on the stream have completed:
    // their flags are final.  Nothing below sets a flag.
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned f = *(volatile unsigned *)&L.scr->status;
        if (f)
            atomicOr(&g_search_fault, f);
    }
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int kmax = L.L_max;
    unsigned char *ws = smem + (threadIdx.x >> 5) * fb_exact_smem_per_warp(kmax);
    unsigned long long *kd = (unsigned long long *)ws + lane;   // [kmax][32]
    int *ki = (int *)(ws + (size_t)kmax * 32 * 8) + lane;       // [kmax][32]
    unsigned nfb = *(volatile unsigned *)&L.scr->n_fallback3;
    if ((long long)nfb > L.fb_cap)
        nfb = (unsigned)L.fb_cap;
    const unsigned long long INF64 = 0x7ff0000000000000ull;
    unsigned long long nfp = 0;
    // one entry per warp, then the queue (as k_tnn_warp)
    unsigned e = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (bool first = true;; first = false) {
        if (!first) {
            if (lane == 0)
                e = atomicAdd(&L.scr->fb_next3, 1u) + gridDim.x * TNN_WARPS_PER_CTA;
            e = __shfl_sync(FULLMASK, e, 0);
        }
        if (e >= nfb)
            break;
        const int2 ent = L.fb_list3[e];
        const KnnWin *W = L.nwin <= 1 ? &L.w0 : L.wins + ent.x;
        const float4 q = W->q[ent.y];
        const QCtx c = make_qctx(W, q, true);
        const float s0 = W->sig[0], s1 = W->sig[1], s2 = W->sig[2], s3 = W->sig[3];
        const float T32 = c.T32;
        const int k = W->k;
        // pass 1: the k-th smallest FP32 key over the valid points (each lane
        // keeps its k smallest, then a k-round warp merge)
        for (int r = 0; r < k; ++r)
            kd[r * 32] = SENT;
        int cnt = 0;
        for (int j = lane; j < W->n; j += 32) {
            const float4 p = W->pts[j];
            if (!(p.w < T32))
                continue;
            const unsigned long long key = pack_key(dist32(c, s0, s1, s2, s3, p), j);
            if (!(key < kd[(k - 1) * 32]))
                continue;
            int pos = cnt < k ? cnt : k - 1;
            while (pos > 0) {
                const unsigned long long pk = kd[(pos - 1) * 32];
                if (pk < key)
                    break;
                kd[pos * 32] = pk;
                --pos;
            }
            kd[pos * 32] = key;
            if (cnt < k)
                ++cnt;
        }
        unsigned long long kth = SENT;
        {
            int h = 0;
            for (int r = 0; r < k; ++r) {
                const unsigned long long v = h < cnt ? kd[h * 32] : SENT;
                unsigned long long mv = v;
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long ov = shfl_xor_u64(mv, o);
                    mv = ov < mv ? ov : mv;
                }
                if (v == mv && h < cnt)
                    ++h;
                kth = mv;
            }
        }
        // Every point of the exact top k has d32 <= tau32 (1 + 2^-20): at
        // least k points have d32 <= tau32, so d64 of the k-th is at most
        // tau32 / (1 - 2^-21), and d32 <= d64 (1 + 2^-21).
        const float tau32 = key_d(kth);
        const float lim = fmaf(tau32, 0x1p-19f, tau32);
        // pass 2: FP64 distances of the points within that bound only
        for (int r = 0; r < k; ++r) {
            kd[r * 32] = INF64;
            ki[r * 32] = 0x7fffffff;
        }
        cnt = 0;
        for (int j = lane; j < W->n; j += 32) {
            const float4 p = W->pts[j];
            if (!(p.w < T32) || !(dist32(c, s0, s1, s2, s3, p) <= lim))
                continue;
            const unsigned long long db =
                (unsigned long long)__double_as_longlong(dist64(W->sigd, q, p));
            nfp++;
            const unsigned long long wd = kd[(k - 1) * 32];
            if (!(db < wd || (db == wd && j < ki[(k - 1) * 32])))
                continue;
            int pos = cnt < k ? cnt : k - 1;
            while (pos > 0) {
                const unsigned long long pd = kd[(pos - 1) * 32];
                const int pi = ki[(pos - 1) * 32];
                if (pd < db || (pd == db && pi < j))
                    break;
                kd[pos * 32] = pd;
                ki[pos * 32] = pi;
                --pos;
            }
            kd[pos * 32] = db;
            ki[pos * 32] = j;
            if (cnt < k)
                ++cnt;
        }
        // merge the 32 lists by (d2, index)
        int h = 0;
        int32_t *oi = W->out_idx + (int64_t)ent.y * k;
        float *od = W->out_d2 + (int64_t)ent.y * k;
        for (int r = 0; r < k; ++r) {
            const unsigned long long vd = h < cnt ? kd[h * 32] : INF64;
            const int vi = h < cnt ? ki[h * 32] : 0x7fffffff;
            unsigned long long md = vd;
            int mi = vi;
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long od_ = __shfl_xor_sync(FULLMASK, md, o);
                const int oi_ = __shfl_xor_sync(FULLMASK, mi, o);
                if (od_ < md || (od_ == md && oi_ < mi)) {
                    md = od_;
                    mi = oi_;
                }
            }
            if (vd == md && vi == mi && h < cnt)
                ++h;
            if (lane == 0) {
                const bool ok = md != INF64;
                oi[r] = ok ? mi : -1;
                od[r] = ok ? (float)__longlong_as_double((long long)md) : INFINITY;
            }
        }
        __syncwarp();
    }
    unsigned long long x = nfp;
    for (int o = 16; o > 0; o >>= 1)
        x += __shfl_xor_sync(FULLMASK, x, o);
    if (lane == 0 && x)
        atomicAdd(&L.scr->stats[4], x);
    if (blockIdx.x == 0 && threadIdx.x == 0)
        L.scr->stats[6] = nfb;
}
