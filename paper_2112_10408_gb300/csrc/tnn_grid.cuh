// TNN search over the time-bucketed spatial grid of the index.
//
// One warp answers a tile of up to 32 queries, one query per lane.  A key of
// the grid (bucket of t_A, cell of the midpoint) has its own lower bound --
// distance from the query to the cell rectangle minus the key's extent, plus
// the temporal part from the key's largest t_B -- which never exceeds the
// cylinder bound of any member segment, so whole keys are excluded at once by
// the exclusion criterion of Sec. 3.4.
//
//   near    the segments of the 3 x 3 cells around the tile in the newest
//           buckets, 32 at a time, one per lane: by ascending bound over the
//           whole tile, as far as some lane's pruning key reaches, every
//           lane's own cylinder bound, and the segment's points if one of
//           them does not exceed its lane's key (Algorithm 2 fetches the
//           nearest first).
//   main    buckets from the causal end backwards; a bucket is visited while
//           the temporal bound of its running maximum of t_B does not exceed
//           some lane's pruning key (Algorithm 2's stop rule); inside it the
//           other cells within reach, the keys whose bound does not exceed a
//           lane's key, and their segments as above.
//
// Points reach the lists 32 at a time.  A lane keeps its candidates as sorted
// 32-bit keys in registers: the upper bits of the FP32 distance above the
// point's slot in a per-tile table.  Every 8 points are sorted by Batcher's
// odd-even merge network and merged with the list by a bitonic network:
// minima and maxima only, no branch, no shared memory, every lane in step.
// At the end the distances of the k + 4 smallest are taken again in full FP32
// and settled as before.
//
// Bound: issue and latency of this arithmetic (data are L2-resident; DRAM
// sees little more than the written lists).  A sorted 64-bit list per lane in
// shared memory, with one insertion per candidate, spent half of the kernel
// in chains of dependent loads and stores at a different moment in every
// lane: 615 us for 400,000 flight samples at k = 32 and 6,774 us for
// 4,000,000; the networks take 284 and 3,088 us, the latency of a single tile
// (10,000 points, k = 8) falls from 170 to 80 us.  The instruction cache sets
// the batch: straight-line code for 32 points a time executes the fewest
// instructions but streams its code (459 us, over half of the stall cycles
// waiting for instructions), 16 take 306 and 8 take 284 us; for the same
// reason everything done once per tile is rolled into short loops.  Bounding a
// segment over the whole tile first, one segment per lane, and per lane only
// when its turn comes (every lane's bound of every staged segment before: 47
// of them per query at 400,000 points), and reading the key records of as many
// buckets as fill a warp took these three figures from 280, 3,016 and 79 us to
// 232, 2,669 and 44 us; bounding the keys the same way, two per lane and round
// of reads, 4,000,000 to 2,497 us; settling only the runs of rows that are not
// certainly in order and keeping the warp's counters and rectangle in shared
// memory (fewer spills, 60 instead of 69 KB of code) to 217, 2,318 and 40 us.
// What that needs to be exact (the farthest of the first k rows, the margin
// beyond a bucket's width) and 64-bit counters cost 0.5 %: 214.4 -> 215.8 and
// 2,349 -> 2,356 us timed in turn, 41.8 on both sides.
// (More rows per step of the settlement, 4, 6 or 9 instead of 2, are slower:
// 234, 247, 257 against 229 us.  Dropping single points by their distance to the
// tile's rectangle before the lanes score them costs more than it saves: 251
// against 234 us.)
#pragma once
#include "tnn_device.cuh"

#ifndef TNN_SEED_BUCKETS
#define TNN_SEED_BUCKETS 3 // newest buckets whose 3 x 3 cells start a tile (at most 3)
#endif

// Lower bound on the cylinder bound (and so on the FP32 distance of any
// valid member) of every segment of one key.
__device__ __forceinline__ float cell_lb(const QCtx &c, float st, float rx0, float rx1,
                                         float ry0, float ry1, float ext, float tBk)
{
    const float dx = fmaxf(fmaxf(rx0 - c.sx, c.sx - rx1), 0.0f);
    const float dy = fmaxf(fmaxf(ry0 - c.sy, c.sy - ry1), 0.0f);
    const float a2 = fmaf(dy, dy, dx * dx);
    const float dist = a2 * rsqrtf(fmaxf(a2, 1e-37f));
    const float sp = fmaxf(fmaf(dist, 1.0f - 0x1p-20f, -(ext + c.delta)), 0.0f);
    const float et = fmaxf(__fsub_rd(c.qt, fminf(tBk, c.T32)), 0.0f);
    return fmaf(sp, sp, (st * et) * et) * (1.0f - 0x1p-19f);
}

// Cells [c0, c1] of one axis (n cells of size 1 / inv_cell from o) whose
// span can come within R of the interval [s0, s1].  The FP32 evaluation of
// the indices here and of the cell corners at query time errs by at most
// 2^-21 ((|s0| + R + 2|o|) inv_cell + n) cells; the slack is twice that plus
// 2^-10.  (A whole cell of margin on each side would triple the cells
// examined at the usual cell sizes, and still fall short for coordinates far
// from the origin.)
__device__ __forceinline__ void reach_cells(float s0, float s1, float R, float o, float inv_cell, int n,
                                            int &c0, int &c1)
{
    const float slack =
        fmaf(0x1p-20f, fmaf(fabsf(s0) + fabsf(s1) + R + 2.0f * fabsf(o), inv_cell, (float)n), 0x1p-10f);
    c0 = max((int)floorf(fmaxf(fmaf(s0 - R - o, inv_cell, -slack), -1.0f)), 0);
    c1 = min((int)floorf(fminf(fmaf(s1 + R - o, inv_cell, slack), (float)n)), n - 1);
}

// Smallest and largest of the warp (NaN only if every lane's is).
__device__ __forceinline__ float warp_minf(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "n"(0xffffffff));
    return r;
}
__device__ __forceinline__ float warp_maxf(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "n"(0xffffffff));
    return r;
}

// Lower bound on seg_lb of one segment over a group of queries whose scaled
// x, y lie in [bx0, bx1] x [by0, by1], whose times are at least qt, whose
// thresholds are at most T32 and lie at least `gap` before them: distance of
// the two rectangles instead of point and line.
struct GroupBox {
    float bx0, bx1, by0, by1, qt, T32, gap, delta;
};
__device__ __forceinline__ float box_lb(const GroupBox &g, float st, float4 a, float4 u, float4 b)
{
    const float ex = a.x + b.x, ey = a.y + b.y;
    const float dx = fmaxf(fmaxf(fminf(a.x, ex) - g.bx1, g.bx0 - fmaxf(a.x, ex)), 0.0f);
    const float dy = fmaxf(fmaxf(fminf(a.y, ey) - g.by1, g.by0 - fmaxf(a.y, ey)), 0.0f);
    const float a2 = fmaf(dy, dy, dx * dx);
    const float dist = a2 * rsqrtf(fmaxf(a2, 1e-37f));
    const float sp = fmaxf(fmaf(dist, 1.0f - 0x1p-20f, -(b.w + g.delta)), 0.0f);
    const float et = fmaxf(fmaxf(__fsub_rd(g.qt, u.w), g.gap), 0.0f);
    const float lb = fmaf(sp, sp, (st * et) * et) * (1.0f - 0x1p-18f);
    return (a.w < g.T32) ? lb : INFINITY;
}

// The same for every segment of one grid key (cell rectangle, extent, largest
// t_B).
__device__ __forceinline__ float box_key_lb(const GroupBox &g, float st, float rx0, float rx1, float ry0,
                                            float ry1, float ext, float tBk)
{
    const float dx = fmaxf(fmaxf(rx0 - g.bx1, g.bx0 - rx1), 0.0f);
    const float dy = fmaxf(fmaxf(ry0 - g.by1, g.by0 - ry1), 0.0f);
    const float a2 = fmaf(dy, dy, dx * dx);
    const float dist = a2 * rsqrtf(fmaxf(a2, 1e-37f));
    const float sp = fmaxf(fmaf(dist, 1.0f - 0x1p-20f, -(ext + g.delta)), 0.0f);
    const float et = fmaxf(fmaxf(__fsub_rd(g.qt, tBk), g.gap), 0.0f);
    return fmaf(sp, sp, (st * et) * et) * (1.0f - 0x1p-18f);
}

// ------------------------------------------------- candidate keys, networks

#define TG_EMPTY 0xffffffffu // sorts after every key
#define TG_INF 0x7f800000u   // keys of infinite distances
#define TG_ROWS 2            // list rows settled per step
#define TG_EXTRA 4           // candidates kept beyond the k-th
#define TG_NB 8        // points sorted at a time
#define TG_INSERT 1    // batches with at most this many candidates are inserted one by one
                       // (400,000 points: 1 279.8 us, 2 280.0, 3 281.3, 5 285.2)
#define TG_KEYS 2         // grid keys per lane and round of reads (4: 227 us against 217)
#define TG_MIN_GROUP 3       // smaller groups of a tile go to the warp-per-query kernel

// Key of a distance (>= 0) in a slot: its bits, the lowest SB replaced by the
// slot.  Keys of one lane order like the distances up to the 2^(SB - 23) that
// the slot displaces.
template <int SB> struct Slots {
    static constexpr int n = 1 << SB;
    static constexpr unsigned mask = n - 1u;
    static __device__ __forceinline__ unsigned key(float d, unsigned s)
    {
        return (__float_as_uint(d) & ~mask) | s;
    }
    // smallest and largest distance a key can stand for
    static __device__ __forceinline__ float lower(unsigned key) { return __uint_as_float(key & ~mask); }
    static __device__ __forceinline__ float upper(unsigned key) { return __uint_as_float(key | mask); }
};
// 512 slots; 1024 for the longest lists, whose tiles hold more points
template <int NL> using TileSlots = Slots<(NL > 32 ? 10 : 9)>;

__device__ __forceinline__ void tg_cmpx(unsigned &a, unsigned &b)
{
    const unsigned lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort (K. E. Batcher, Sorting networks and their
// applications, 1968): comparators of round (P, K).
template <int N, int P, int K> __device__ __forceinline__ void tg_sort_round(unsigned (&v)[N])
{
#pragma unroll
    for (int x = K % P; x + K < N; ++x)
        if ((x - K % P) % (2 * K) < K && x / (2 * P) == (x + K) / (2 * P))
            tg_cmpx(v[x], v[x + K]);
    if constexpr (K > 1)
        tg_sort_round<N, P, K / 2>(v);
}
template <int N, int P = 1> __device__ __forceinline__ void tg_sort(unsigned (&v)[N])
{
    tg_sort_round<N, P, P>(v);
    if constexpr (2 * P < N)
        tg_sort<N, 2 * P>(v);
}
// Ascending order of a bitonic sequence.
template <int N, int H = N / 2> __device__ __forceinline__ void tg_bitonic(unsigned (&v)[N])
{
#pragma unroll
    for (int x = 0; x < N; ++x)
        if ((x & H) == 0)
            tg_cmpx(v[x], v[x + H]);
    if constexpr (H > 1)
        tg_bitonic<N, H / 2>(v);
}
// First H values of a bitonic sequence of 2 H: its H smallest, bitonic again.
template <int N, int H = N / 2> __device__ __forceinline__ void tg_smallest4(unsigned (&v)[N])
{
#pragma unroll
    for (int x = 0; x < H; ++x)
        v[x] = min(v[x], v[x + H]);
    if constexpr (H > TG_EXTRA)
        tg_smallest4<N, H / 2>(v);
}

// Merge the sorted batch b into the sorted list a (the NL smallest keys stay)
// and what leaves it into the TG_EXTRA next ones o.
template <int NL, int NB>
__device__ __forceinline__ void tg_merge(unsigned (&a)[NL], unsigned (&o)[TG_EXTRA], const unsigned (&b)[NB])
{
    unsigned r[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const unsigned x = a[NL - NB + i], y = b[NB - 1 - i];
        a[NL - NB + i] = min(x, y);
        r[i] = max(x, y);
    }
    tg_bitonic<NL>(a);
    tg_smallest4<NB>(r);
    unsigned e[TG_EXTRA];
#pragma unroll
    for (int i = 0; i < TG_EXTRA; ++i)
        e[i] = r[i];
    tg_bitonic<TG_EXTRA>(e);
#pragma unroll
    for (int i = 0; i < TG_EXTRA; ++i)
        o[i] = min(o[i], e[TG_EXTRA - 1 - i]);
    tg_bitonic<TG_EXTRA>(o);
}

template <int NL>
__device__ __forceinline__ void tg_insert(unsigned (&a)[NL], unsigned (&o)[TG_EXTRA], unsigned key)
{
#pragma unroll
    for (int i = 0; i < NL; ++i) {
        const unsigned t = min(a[i], key);
        key = max(a[i], key);
        a[i] = t;
    }
#pragma unroll
    for (int i = 0; i < TG_EXTRA; ++i) {
        const unsigned t = min(o[i], key);
        key = max(o[i], key);
        o[i] = t;
    }
}

// ------------------------------------------------------------ shared memory

// Per warp.  While points are gathered: the batch's points, staged segments,
// the slots in use and their prefix, the key ranges' ends and offsets; the
// slot table behind them.  To
// settle, the lists' 32-bit keys take the first part's place, and then the
// 64-bit lists [NL + TG_EXTRA][32] everything's.
template <int NL> struct TileSmem {
    union {
        struct {
            float4 pts[32];
            float4 seg[32][3];
            unsigned used[32]; // one word per 32 slots
            int pre[32];
            int kend[32 * TG_KEYS];
            int krel[32 * TG_KEYS];
        };
        unsigned raw[NL + TG_EXTRA][32];
    };
    int slot[TileSlots<NL>::n];
};

// Kept through all of it: the group's rectangle and the warp's counters
// (queries, bounds, distances, segments, FP64 distances), which would take
// registers from the lists.  A warp can take more than 2^32 distances.
struct TileKeep {
    GroupBox box;
    unsigned long long count[6];
};

template <int NL> __host__ __device__ constexpr size_t tg_smem_per_warp()
{
    const size_t lists = (size_t)(NL + TG_EXTRA) * 256;
    return (lists > sizeof(TileSmem<NL>) ? lists : sizeof(TileSmem<NL>)) + sizeof(TileKeep);
}

// Entry e of a lane's settled list: the lane's column is rotated by the entry
// so that both a column (settlement) and a row (output) are read without bank
// conflicts.
__device__ __forceinline__ unsigned long long *tg_entry(unsigned long long *Kw, int e, int lane)
{
    return Kw + e * 32 + (lane ^ (e & 31));
}

// Settle rows r0 .. r1 of one query's list, whose order is not certain: sort
// them by their exact keys, then rank chains of close ones in FP64, in place.
// The rows before and after are certain.  Bit 0 of the result: settled; the
// rest counts the FP64 distances.  Out of line: a few per cent of the queries
// come here, mostly with two rows.
static __device__ __noinline__ unsigned tg_settle(const KnnWin *W, float4 q, unsigned long long *Kw,
                                                  int lane, int r0, int r1)
{
    for (int i = r0 + 1; i <= r1; ++i) {
        const unsigned long long v = *tg_entry(Kw, i, lane);
        int j = i;
        while (j > r0) {
            const unsigned long long u = *tg_entry(Kw, j - 1, lane);
            if (u <= v)
                break;
            *tg_entry(Kw, j, lane) = u;
            --j;
        }
        if (j < i)
            *tg_entry(Kw, j, lane) = v;
    }
    const bool exact_all = (W->flags & TNN_FLAG_EXACT_D2) != 0;
    unsigned nfp = 0;
    int i = r0;
    while (i <= r1) {
        const unsigned long long ki = *tg_entry(Kw, i, lane);
        if (ki == SENT)
            break;
        int e = i;
        float de = key_d(ki);
        while (e < r1) {
            const unsigned long long kn = *tg_entry(Kw, e + 1, lane);
            const float dn = key_d(kn);
            if (kn == SENT || !(dn <= fmaf(de, 0x1p-17f, de) + 0x1p-100f))
                break;
            ++e;
            de = dn;
        }
        const int c = e - i + 1;
        if (c > CMAX)
            return nfp << 1;
        if (c > 1 || exact_all) {
            double dd[CMAX];
            int id[CMAX];
            for (int t = 0; t < c; ++t) {
                const int j = key_i(*tg_entry(Kw, i + t, lane));
                const double d = dist64(W->sigd, q, W->pts[j]);
                ++nfp;
                int pos = t;
                while (pos > 0 && (dd[pos - 1] > d || (dd[pos - 1] == d && id[pos - 1] > j))) {
                    dd[pos] = dd[pos - 1];
                    id[pos] = id[pos - 1];
                    --pos;
                }
                dd[pos] = d;
                id[pos] = j;
            }
            for (int t = 0; t < c; ++t)
                *tg_entry(Kw, i + t, lane) = pack_key((float)dd[t], id[t]);
        }
        i = e + 1;
    }
    return (nfp << 1) | 1u;
}

// Cells of the newest buckets in the order they are staged: the tile's own
// first, then its neighbours, by bucket age.  db * 16 + (dy + 1) * 4 + dx + 1.
static __device__ const unsigned char tg_seed_cell[32] = {
    5,  21, 4,  6,  1,  9,  20, 22, 17, 25, 0,  2,  8,  10, 16, 18, 24, 26, 37, 36, 38, 33, 41, 32, 34, 40, 42,
    0,  0,  0,  0,  0};

// CTAs per SM: the list's registers (list + batch) set it.  400,000 points, k
// = 32: 3 CTAs 244.5 us, 4 234.2, 5 263.2 (spills); 10,000 points, k = 8: 5
// 41.5, 6 43.6; mixed windows with k = 64: 2 1,311, 3 1,304, 4 1,391.
template <int NL> struct TileCtas {
    static constexpr int value = NL == 64 ? 3 : NL == 32 ? 4 : 5;
};

// The grid-order tile kernel for k <= NL.  A list shorter than NL keys holds
// zeros in front (they never leave and are skipped at the end), so that its
// last key is the k-th smallest.
template <int NL>
__global__ void __launch_bounds__(TNN_WARPS_PER_CTA * 32, TileCtas<NL>::value)
    k_tnn_grid_search(const __grid_constant__ KnnLaunch L)
{
    using SL = TileSlots<NL>;
    constexpr int NB = NL < TG_NB ? NL : TG_NB; // points per network batch
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    unsigned char *ws = smem + (threadIdx.x >> 5) * tg_smem_per_warp<NL>();
    TileSmem<NL> &S = *(TileSmem<NL> *)ws;
    unsigned long long *Kw = (unsigned long long *)ws;
    TileKeep &KP = *(TileKeep *)(ws + tg_smem_per_warp<NL>() - sizeof(TileKeep));
    if (lane < 6)
        KP.count[lane] = 0;
    __syncwarp();
    pdl_trigger();

    // First tile by the warp's number, then the queue.
    long long claim = (long long)blockIdx.x * TNN_WARPS_PER_CTA + (threadIdx.x >> 5);
    for (;;) {
        const long long tile = L.tile_lo + __shfl_sync(FULLMASK, claim, 0);
        if (tile >= L.total_tiles)
            break;
        const KnnWin *W = find_window(L, tile);
        int64_t qrow;
        const bool active = tile_query(W, tile, lane, qrow);
        const float4 q = active ? W->q[qrow] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float s0 = W->sig[0], s1 = W->sig[1], s2 = W->sig[2], s3 = W->sig[3];
        const float4 *__restrict__ pts = W->pts;
        const GridDesc &G = W->grid;
        const float tau_defer = W->tau_defer;
        const int k = W->k;

        // A tile whose queries lie far apart (the caller's own order, two
        // flights in one tile) is answered in groups around its first query
        // not yet taken; lanes of tiny groups get a warp of their own.
        unsigned todo = __ballot_sync(FULLMASK, active);
        unsigned lone = 0;
        while (todo) {
        unsigned grp = todo;
        if (tau_defer < INFINITY) {
            const int ld = __ffs(todo) - 1;
            const float gx = W->ssq[0] * q.x, gy = W->ssq[1] * q.y;
            const float lx = __shfl_sync(FULLMASK, gx, ld), ly = __shfl_sync(FULLMASK, gy, ld);
            const float lt = __shfl_sync(FULLMASK, q.w, ld);
            const bool near = fabsf(gx - lx) <= 1.5f * G.cell && fabsf(gy - ly) <= 1.5f * G.cell &&
                              fabsf(q.w - lt) <= 1.5f * G.dt;
            grp = __ballot_sync(FULLMASK, near) & todo;
            grp |= 1u << ld;
            todo &= ~grp;
            if (__popc(grp) < TG_MIN_GROUP) {
                lone |= grp;
                continue;
            }
        } else {
            todo = 0;
        }
        const bool act = (grp >> lane) & 1u;
        const QCtx c = make_qctx(W, q, act);

        const float tmax = warp_maxf(c.T32);
        const float bx0 = warp_minf(act ? c.sx : INFINITY);
        const float bx1 = warp_maxf(act ? c.sx : -INFINITY);
        const float by0 = warp_minf(act ? c.sy : INFINITY);
        const float by1 = warp_maxf(act ? c.sy : -INFINITY);
        {
            const GroupBox box = {bx0, bx1, by0, by1, warp_minf(act ? c.qt : INFINITY), tmax,
                                  warp_minf(act ? __fsub_rd(c.qt, c.T32) : INFINITY),
                                  warp_maxf(act ? c.delta : 0.0f)};
            __syncwarp();
            if (lane == 0) {
                KP.box = box;
                KP.count[0] += __popc(grp);
            }
            __syncwarp();
        }
        int bhi = -1;
        {
            const float fb = (tmax - G.t0) * G.inv_dt;
            if (fb >= 0.0f)
                bhi = (int)fminf(floorf(fb), (float)(G.nb - 1));
        }
        const int hx = min(max((int)floorf((0.5f * (bx0 + bx1) - G.x0) * G.inv_cell), 0), G.nx - 1);
        const int hy = min(max((int)floorf((0.5f * (by0 + by1) - G.y0) * G.inv_cell), 0), G.ny - 1);

        unsigned a[NL], o[TG_EXTRA];
#pragma unroll
        for (int i = 0; i < NL; ++i)
            a[i] = i < NL - k ? 0u : TG_EMPTY;
#pragma unroll
        for (int i = 0; i < TG_EXTRA; ++i)
            o[i] = TG_EMPTY;
        // Pruning key: points above it are not needed.  A little above the
        // k-th key so that every point its FP64 settlement may involve is seen.
        float tau = INFINITY;
        // what a segment's bound is compared with in the present phase
        float lim = act ? tau_defer : -1.0f;
        bool given_up = false; // more distinct candidates than slots (warp-uniform)
        bool deferred = false;

        int base = 0, fill = 0, myidx = 0; // next slot; points gathered so far, this lane's
        // main phase: next bucket, buckets of the present group, their cells
        int b = bhi, gb = 0, t0 = 0, ncells = 0, cx0 = 0, cy0 = 0, wx = 1, nc = 1;
        bool near_phase = true;
        int total = 0, pos = 0; // segments of the present key group, handled so far

        // The segments of up to 32 TG_KEYS keys (lane: [klo, klo + kn) in key
        // order) become the present group.
        auto take_keys = [&](const int (&klo)[TG_KEYS], const int (&kn)[TG_KEYS]) {
            int inc = 0;
#pragma unroll
            for (int u = 0; u < TG_KEYS; ++u)
                inc += kn[u];
            int at = -inc;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const int v = __shfl_up_sync(FULLMASK, inc, s);
                if (lane >= s)
                    inc += v;
            }
            at += inc;
            __syncwarp();
#pragma unroll
            for (int u = 0; u < TG_KEYS; ++u) {
                S.krel[lane * TG_KEYS + u] = klo[u] - at; // record = krel[j] + position in the group
                at += kn[u];
                S.kend[lane * TG_KEYS + u] = at;
            }
            total = __shfl_sync(FULLMASK, inc, 31);
            pos = 0;
            __syncwarp();
        };
        {
            const int seed_cell = tg_seed_cell[lane];
            const int bq = bhi - (seed_cell >> 4);
            const int cx = hx + (seed_cell & 3) - 1, cy = hy + ((seed_cell >> 2) & 3) - 1;
            int klo[TG_KEYS] = {0}, kn[TG_KEYS] = {0};
            if (lane < 9 * TNN_SEED_BUCKETS && bq >= 0 && cx >= 0 && cx < G.nx && cy >= 0 && cy < G.ny) {
                const int key = bq * G.ncell + cy * G.nx + cx;
                klo[0] = __ldg(G.off + key);
                kn[0] = __ldg(G.off + key + 1) - klo[0];
            }
            take_keys(klo, kn);
        }

        for (;;) {
            const int cnt = min(32, total - pos);
            bool flush = false;
            if (cnt <= 0) {
                // the group is done: next one, or first what is gathered
                if (near_phase) {
                    if (fill > 0) {
                        flush = true;
                    } else {
                        // a lane whose key is still above the deferral
                        // threshold (far neighbours, or a list not yet full)
                        // would make the whole tile visit a wide region
                        near_phase = false;
                        deferred = act && !(tau <= tau_defer);
                        continue;
                    }
                } else if (t0 >= ncells) {
                    if (fill > 0) {
                        flush = true;
                    } else {
                        // the next buckets, as many as give 32 TG_KEYS cells:
                        // their records are one round of reads
                        b -= gb;
                        if (b < 0)
                            break;
                        const float bp = __ldg(G.bpm + max(b - lane, 0));
                        const float tl = time_lb(c, s3, __shfl_sync(FULLMASK, bp, 0));
                        const bool done = !act || deferred || !(tl <= tau);
                        if (__all_sync(FULLMASK, done))
                            break;
                        lim = done ? -1.0f : tau;
                        const float tmx = warp_maxf(done ? 0.0f : tau);
                        int cx1 = G.nx - 1, cy1 = G.ny - 1;
                        cx0 = 0;
                        cy0 = 0;
                        if (tmx < INFINITY) {
                            // any key outside this reach has a bound above every key
                            const float R = sqrtf(tmx) * (1.0f + 0x1p-18f) + __ldg(G.ext_max) + KP.box.delta;
                            reach_cells(KP.box.bx0, KP.box.bx1, R, G.x0, G.inv_cell, G.nx, cx0, cx1);
                            reach_cells(KP.box.by0, KP.box.by1, R, G.y0, G.inv_cell, G.ny, cy0, cy1);
                        }
                        wx = cx1 - cx0 + 1;
                        nc = max(wx, 0) * max(cy1 - cy0 + 1, 0);
                        if (nc == 0)
                            break; // no cell within reach
                        const int most = min(min(b + 1, 32), 32 * TG_KEYS / nc);
#pragma unroll 1
                        for (gb = 1; gb < most; ++gb) {
                            const float tg = time_lb(c, s3, __shfl_sync(FULLMASK, bp, gb));
                            if (!__any_sync(FULLMASK, !done && tg <= tau))
                                break;
                        }
                        ncells = nc * gb;
                        t0 = 0;
                        continue;
                    }
                } else {
                    // up to 32 TG_KEYS cells of the group: the keys the
                    // query group as a whole may need
                    const float inv_nc = 1.0f / (float)nc, inv_wx = 1.0f / (float)wx, reach = warp_maxf(lim);
                    int klo[TG_KEYS], kn[TG_KEYS], any = 0;
                    int4 kr[TG_KEYS];
                    int kx[TG_KEYS], ky[TG_KEYS];
#pragma unroll
                    for (int u = 0; u < TG_KEYS; ++u) {
                        const int t = t0 + u * 32 + lane;
                        // quotients of integers below 2^21: exact
                        const int db = (int)(((float)t + 0.5f) * inv_nc), rem = t - db * nc;
                        const int dy = (int)(((float)rem + 0.5f) * inv_wx);
                        kx[u] = cx0 + rem - dy * wx;
                        ky[u] = cy0 + dy;
                        const bool staged = b - db > bhi - TNN_SEED_BUCKETS && abs(kx[u] - hx) <= 1 &&
                                            abs(ky[u] - hy) <= 1;
                        kr[u] = t < ncells && !staged ? __ldg(G.krec + ((b - db) * G.ncell + ky[u] * G.nx + kx[u]))
                                                      : make_int4(0, 0, 0, 0);
                    }
#pragma unroll
                    for (int u = 0; u < TG_KEYS; ++u) {
                        const float rx0 = G.x0 + (float)kx[u] * G.cell, ry0 = G.y0 + (float)ky[u] * G.cell;
                        const bool want = box_key_lb(KP.box, s3, rx0, rx0 + G.cell, ry0, ry0 + G.cell,
                                                     __int_as_float(kr[u].z), __int_as_float(kr[u].w)) <= reach;
                        klo[u] = kr[u].x;
                        kn[u] = want ? kr[u].y - kr[u].x : 0;
                        any |= kn[u];
                    }
                    t0 += 32 * TG_KEYS;
                    if (__any_sync(FULLMASK, any != 0))
                        take_keys(klo, kn);
                    continue;
                }
            }

            // ---- the next (up to 32) segments of the key group, one per lane,
            // by their bound over the whole query group
            int sfirst = 0, scnt = 0;
            unsigned score = TG_EMPTY; // that bound above the lane
            if (cnt > 0) {
                __syncwarp();
                if (lane < cnt) {
                    const int g = pos + lane;
                    int lo = 0, hi = 32 * TG_KEYS - 1; // smallest key with kend > g
#pragma unroll 1
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (S.kend[mid] > g)
                            hi = mid;
                        else
                            lo = mid + 1;
                    }
                    const float4 *r = G.gseg + 4 * (size_t)(S.krel[lo] + g);
                    const float4 ra = __ldg(r), ru = __ldg(r + 1), rb = __ldg(r + 2), r3 = __ldg(r + 3);
                    S.seg[lane][0] = ra;
                    S.seg[lane][1] = ru;
                    S.seg[lane][2] = rb;
                    sfirst = __float_as_int(r3.x);
                    scnt = __float_as_int(r3.y);
                    const float lb = box_lb(KP.box, s3, ra, ru, rb);
                    if (lb < INFINITY) // truncated towards zero: still a bound
                        score = (__float_as_uint(lb) & ~31u) | (unsigned)lane;
                }
                pos += cnt;
                __syncwarp();
            }

            // ---- their points, 32 at a time: nearest segments first, while
            // some query's own bound allows
            int lf = 0, lc = 0; // points left of the segment taken last
            float most = warp_maxf(lim);
            for (;;) {
                while (fill < 32) {
                    if (lc == 0) {
                        const unsigned best = __reduce_min_sync(FULLMASK, score);
                        if (best == TG_EMPTY || !(__uint_as_float(best & ~31u) <= most))
                            break;
                        const int j = best & 31u;
                        if (lane == j)
                            score = TG_EMPTY;
                        const float lb = seg_lb(c, s3, S.seg[j][0], S.seg[j][1], S.seg[j][2]);
                        if (lane == 0)
                            KP.count[1] += __popc(grp);
                        if (!__any_sync(FULLMASK, lb <= lim))
                            continue;
                        lf = __shfl_sync(FULLMASK, sfirst, j);
                        lc = __shfl_sync(FULLMASK, scnt, j);
                        if (lane == 0)
                            KP.count[3] += __popc(grp);
                    }
                    const int take = min(lc, 32 - fill);
                    if (lane >= fill && lane < fill + take)
                        myidx = lf + lc - 1 - (lane - fill); // newest member first
                    lc -= take;
                    fill += take;
                }
                if (fill == 0 || (fill < 32 && !flush))
                    break;
                if (base > SL::n - 32) {
                    // renumber the slots that some list still holds
                    __syncwarp();
                    S.used[lane] = 0;
                    __syncwarp();
                    unsigned t[NL + TG_EXTRA]; // in local memory: this is rare
#pragma unroll
                    for (int i = 0; i < NL; ++i)
                        t[i] = a[i];
#pragma unroll
                    for (int i = 0; i < TG_EXTRA; ++i)
                        t[NL + i] = o[i];
#pragma unroll 1
                    for (int i = 0; i < NL + TG_EXTRA; ++i)
                        if (t[i] != TG_EMPTY)
                            atomicOr(&S.used[(t[i] & SL::mask) >> 5], 1u << (t[i] & 31u));
                    __syncwarp();
                    const unsigned u = S.used[lane];
                    int inc = __popc(u);
#pragma unroll
                    for (int s = 1; s < 32; s <<= 1) {
                        const int v = __shfl_up_sync(FULLMASK, inc, s);
                        if (lane >= s)
                            inc += v;
                    }
                    S.pre[lane] = inc - __popc(u);
                    base = __shfl_sync(FULLMASK, inc, 31);
                    __syncwarp();
#pragma unroll 1
                    for (int i = 0; i < NL + TG_EXTRA; ++i) {
                        const unsigned v = t[i], s = v & SL::mask;
                        if (v != TG_EMPTY)
                            t[i] = (v & ~SL::mask) |
                                   (unsigned)(S.pre[s >> 5] + __popc(S.used[s >> 5] & ((1u << (s & 31u)) - 1u)));
                    }
#pragma unroll
                    for (int i = 0; i < NL; ++i)
                        a[i] = t[i];
#pragma unroll
                    for (int i = 0; i < TG_EXTRA; ++i)
                        o[i] = t[NL + i];
#pragma unroll 1
                    for (int w = 0; w < SL::n / 32; ++w) {
                        const unsigned uw = S.used[w];
                        const int id = S.slot[w * 32 + lane];
                        __syncwarp();
                        if ((uw >> lane) & 1u)
                            S.slot[S.pre[w] + __popc(uw & ((1u << lane) - 1u))] = id;
                        __syncwarp();
                    }
                    if (base > SL::n - 32) {
                        given_up = true;
                        break;
                    }
                }
                __syncwarp();
                {
                    const bool have = lane < fill;
                    float4 p = make_float4(0.f, 0.f, 0.f, INFINITY); // never causal
                    if (have) {
                        p = __ldg(pts + myidx);
                        S.slot[base + lane] = myidx;
                    }
                    S.pts[lane] = p;
                }
                __syncwarp();
                if (lane == 0)
                    KP.count[2] += __popc(grp) * fill;
                if (L.dbg_seen && act)
#pragma unroll 1
                    for (int i = 0; i < fill; ++i)
                        dbg_mark_seen(L, qrow, S.slot[base + i], 1);
                unsigned kept = 0;
#pragma unroll 1
                for (int s = 0; s < fill; s += NB) {
                    unsigned v[NB], mine = 0;
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const float4 p = S.pts[s + i];
                        const float d = dist32(c, s0, s1, s2, s3, p);
                        const bool in = p.w < c.T32 && d <= tau;
                        v[i] = in ? SL::key(d, (unsigned)(base + s + i)) : TG_EMPTY;
                        mine |= in ? 1u << i : 0u;
                    }
                    unsigned any = __reduce_or_sync(FULLMASK, mine);
                    if (!any)
                        continue;
                    kept = 1;
                    if (__popc(any) <= TG_INSERT) {
#pragma unroll 1
                        while (any) {
                            const int i = __ffs(any) - 1;
                            any &= any - 1;
                            const float4 p = S.pts[s + i];
                            const float d = dist32(c, s0, s1, s2, s3, p);
                            const unsigned key = (mine >> i) & 1u ? SL::key(d, (unsigned)(base + s + i)) : TG_EMPTY;
                            tg_insert<NL>(a, o, key);
                        }
                    } else {
                        tg_sort<NB>(v);
                        tg_merge<NL, NB>(a, o, v);
                    }
                    if (a[NL - 1] < TG_INF)
                        tau = fmaf(SL::upper(a[NL - 1]), 0x1p-12f, SL::upper(a[NL - 1])) + 0x1p-98f;
                    lim = fminf(lim, tau);
                }
                base += kept ? 32 : 0;
                fill = 0;
                most = warp_maxf(lim);
            }
            if (given_up)
                break;
        }

        // ---- hand-over of deferred lanes, with a pruning key when k +
        // TG_EXTRA points lie at or below it (and it is a distance: what lies
        // above the key of an overflowed one is no number)
        if (given_up)
            deferred = act;
        if (deferred) {
            const float hand = !given_up && o[TG_EXTRA - 1] < TG_INF
                                   ? SL::upper(o[TG_EXTRA - 1])
                                   : INFINITY;
            const unsigned slot = atomicAdd(&L.scr->n_fallback, 1u);
            if (slot < (unsigned long long)L.fb_cap) {
                L.fb_list[slot] = make_int2(window_id(L, W), (int)qrow);
                L.fb_tau[slot] = hand;
            } else
                atomicOr(&L.scr->status, 1u);
        }

        // ---- settle: exact keys of the k + TG_EXTRA smallest.  Every point
        // outside them lies at or above `bound`.
        const bool settle = act && !deferred;
        float bound = INFINITY;
        bool ok = a[NL - 1] < TG_INF || a[NL - 1] == TG_EMPTY; // else distances overflowed
        if (a[NL - 1] < TG_INF)
            bound = o[TG_EXTRA - 1] != TG_EMPTY ? fminf(SL::lower(o[TG_EXTRA - 1]), tau) : tau;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NL; ++i)
            S.raw[i][lane] = a[i];
#pragma unroll
        for (int i = 0; i < TG_EXTRA; ++i)
            S.raw[NL + i][lane] = o[i];
        // slots to point indices (each lane its own column)
        const int z = NL - k; // rows below hold the leading zeros
#pragma unroll 4
        for (int e = z; e < NL + TG_EXTRA; ++e) {
            const unsigned v = S.raw[e][lane];
            S.raw[e][lane] = settle && v != TG_EMPTY ? (unsigned)S.slot[v & SL::mask] : TG_EMPTY;
        }
        {
            // Exact keys, TG_ROWS rows per step (their gathers in flight
            // together) from the last one down: 64-bit row e covers 32-bit
            // rows 2 e and 2 e + 1, which every lane has read by then.  Rows
            // r0 .. r1 hold every row that is not certainly below its
            // successor: nearer to it than the width of a bucket of truncated
            // keys (at most 2^-23 n of the distance) plus the settlement's
            // margin of 2^-17.  The width, because rows behind the successor
            // may lie lower in its bucket, and rows of r0 .. r1 higher in that
            // of r1; 2^-21 more covers the products of these factors.
            constexpr float link = 0x1p-23f * (float)SL::n + 0x1.1p-17f;
            int r0 = NL + TG_EXTRA, r1 = -1;
            float dn = INFINITY, dk = 0.0f; // dk: the largest of the first k rows
#pragma unroll 1
            for (int e = NL + TG_EXTRA - 1; e >= z; e -= TG_ROWS) {
                unsigned id[TG_ROWS];
                float4 p[TG_ROWS];
#pragma unroll
                for (int u = 0; u < TG_ROWS; ++u)
                    id[u] = S.raw[max(e - u, z)][lane];
                __syncwarp();
#pragma unroll
                for (int u = 0; u < TG_ROWS; ++u)
                    p[u] = __ldg(pts + (id[u] != TG_EMPTY ? id[u] : 0u));
#pragma unroll
                for (int u = 0; u < TG_ROWS; ++u) {
                    const float d = id[u] != TG_EMPTY ? dist32(c, s0, s1, s2, s3, p[u]) : INFINITY;
                    if (e - u >= z) {
                        *tg_entry(Kw, e - u, lane) = pack_key(d, (int)id[u]); // (infinity, -1) is SENT
                        if (dn < fmaf(d, link, d) + 0x1p-99f) {
                            r0 = e - u;
                            r1 = max(r1, e - u + 1);
                        }
                        dn = d;
                        if (e - u < NL)
                            dk = fmaxf(dk, d);
                    }
                }
            }
            // every point outside the list lies at or above `bound`: certainly
            // beyond k listed ones when it is beyond the first k rows, whichever
            // of them is the farthest (a bucket's rows stand in any order)
            ok = ok && !(bound < fmaf(dk, 0x1.1p-17f, dk) + 0x1p-99f);
            // Fewer than k points, perhaps of overflowed distances: these are
            // equal in FP32 and ranked in FP64.
            if ((W->flags & TNN_FLAG_EXACT_D2) || !(dk < INFINITY)) {
                r0 = z;
                r1 = NL + TG_EXTRA - 1;
            }
            if (settle && ok && r0 < r1) {
                const unsigned r = tg_settle(W, q, Kw, lane, r0, r1);
                ok = r & 1u;
                atomicAdd(&KP.count[4], (unsigned long long)(r >> 1));
            }
        }
        if (settle && !ok) {
            const unsigned slot = atomicAdd(&L.scr->n_fallback, 1u);
            if (slot < (unsigned long long)L.fb_cap) // unsettled: -1 - window
                L.fb_list[slot] = make_int2(-1 - window_id(L, W), (int)qrow);
            else
                atomicOr(&L.scr->status, 1u);
        }
        // ---- write the settled rows: consecutive words across the lanes (a
        // store per lane of its own row would touch 32 lines), to the mapped
        // host lists when the call has them
        const unsigned wmask = __ballot_sync(FULLMASK, settle && ok);
        if (wmask) {
            const int64_t off0 = __shfl_sync(FULLMASK, qrow, 0) * k;
            int32_t *oi = (L.mirror_idx ? L.mirror_idx : W->out_idx) + off0;
            float *od = (L.mirror_d2 ? L.mirror_d2 : W->out_d2) + off0;
            if (((k & 3) | (int)(((uintptr_t)oi | (uintptr_t)od) & 15)) == 0) {
                const int kq = k >> 2;
                int row = lane / kq, e = lane % kq;
                const int drow = 32 / kq, de = 32 % kq;
                while (row < 32) {
                    if ((wmask >> row) & 1u) {
                        int ri[4];
                        float rd[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const unsigned long long key = *tg_entry(Kw, z + 4 * e + u, row);
                            ri[u] = key == SENT ? -1 : key_i(key);
                            rd[u] = key == SENT ? INFINITY : key_d(key);
                        }
                        const int64_t w = (int64_t)row * kq + e;
                        ((int4 *)oi)[w] = make_int4(ri[0], ri[1], ri[2], ri[3]);
                        ((float4 *)od)[w] = make_float4(rd[0], rd[1], rd[2], rd[3]);
                    }
                    row += drow;
                    e += de;
                    if (e >= kq) {
                        e -= kq;
                        ++row;
                    }
                }
            } else {
                int row = lane / k, e = lane % k;
                const int drow = 32 / k, de = 32 % k;
                while (row < 32) {
                    if ((wmask >> row) & 1u) {
                        const unsigned long long key = *tg_entry(Kw, z + e, row);
                        oi[(int64_t)row * k + e] = key == SENT ? -1 : key_i(key);
                        od[(int64_t)row * k + e] = key == SENT ? INFINITY : key_d(key);
                    }
                    row += drow;
                    e += de;
                    if (e >= k) {
                        e -= k;
                        ++row;
                    }
                }
            }
        }
        __syncwarp();
        }
        if (lane == 0 && lone)
            KP.count[0] += __popc(lone);
        if (lane == 0)
            claim = (long long)gridDim.x * TNN_WARPS_PER_CTA +
                    (long long)atomicAdd(&L.scr->tile_counter[L.queue], 1ull);
        if ((lone >> lane) & 1u) {
            const unsigned slot = atomicAdd(&L.scr->n_fallback, 1u);
            if (slot < (unsigned long long)L.fb_cap) {
                L.fb_list[slot] = make_int2(window_id(L, W), (int)qrow);
                L.fb_tau[slot] = INFINITY;
            } else
                atomicOr(&L.scr->status, 1u);
        }
        __syncwarp();
    }
    __syncwarp();
    if (lane < 5 && KP.count[lane])
        atomicAdd(&L.scr->stats[lane], KP.count[lane]);
}
