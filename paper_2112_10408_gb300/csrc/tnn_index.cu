// Index construction: Sec. 3.4 (partitioning trajectories into sets of K
// points approximated by segments, the approximation error) and the segment
// matrices A, t_A, B, t_B, U, E of the Fig. 2 caption.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "tnn_internal.cuh"

namespace cg = cooperative_groups;

// ------------------------------------------------------------------ errors

static thread_local char g_err[512];

void tnn_set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

void tnn_clear_error() { g_err[0] = 0; }

extern "C" const char *tnn_last_error(void) { return g_err; }

extern "C" const char *tnn_status_string(tnn_status s)
{
    switch (s) {
    case TNN_OK: return "ok";
    case TNN_ERR_INVALID_ARG: return "invalid argument";
    case TNN_ERR_OOM: return "out of device memory";
    case TNN_ERR_CUDA: return "CUDA error";
    case TNN_ERR_TIMEOUT: return "device wait timed out";
    case TNN_ERR_UNSUPPORTED: return "unsupported";
    }
    return "unknown status";
}

// ----------------------------------------------------------- device helpers

// Order-preserving map of a float to uint32 (negative values included).
__device__ __forceinline__ uint32_t f2ord(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

enum { BAD_VALUE = 1, BAD_ORDER = 2 };

// Words of the build's device header: filled by k_validate and the segment
// fit, read back once.
enum {
    META_FLAG = 0,  // BAD_* bits
    META_CMAX = 1,  // largest |scaled spatial coordinate|, bits
    META_BBOX = 2,  // per axis x, y, z, t: ordered minimum, maximum
    META_DUR = 10,  // summed duration of the K-point sets (a double)
    META_READ = 12, // words the host reads
    META_RMAX = 12, // largest segment radius, bits
    META_EXT = 13,  // largest key extent, bits
    META_WORDS = 16
};

#define VAL_THREADS 256

// One pass over the caller's points by the first `pblocks` blocks: copied
// into the index, every coordinate finite with |v| <= 1e15 (so every FP32
// squared difference stays finite), the largest |sqrt(sigma) x| over the
// spatial axes, the bounding box.  The other blocks take a trajectory per
// warp: times non-decreasing inside it, the summed duration t_last - t_first
// of its K-point sets, which sizes the grid's time buckets, and the sets'
// (first point, count, trajectory) and t_A sort keys.
// (A copy and three kernels before; bound by the reads and the launch.)
__global__ void __launch_bounds__(VAL_THREADS)
    k_validate(const float4 *__restrict__ in, float4 *__restrict__ out, int n, float s0, float s1, float s2,
               const int32_t *__restrict__ traj_off, const int32_t *__restrict__ seg_off, int n_traj, int K,
               int pblocks, int S, int S2, int4 *__restrict__ range, unsigned long long *__restrict__ keys,
               unsigned int *__restrict__ meta)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if ((int)blockIdx.x >= pblocks) {
        // the sort's padding (32 times the trajectories can pass 2^31)
        for (int64_t i = S + (int64_t)(blockIdx.x - pblocks) * VAL_THREADS + threadIdx.x; i < S2;
             i += (int64_t)(gridDim.x - pblocks) * VAL_THREADS)
            keys[i] = ~0ull;
        const int tr = ((int)blockIdx.x - pblocks) * (VAL_THREADS / 32) + w;
        if (tr >= n_traj) // the same for the whole warp
            return;
        const int b = traj_off[tr], e = traj_off[tr + 1];
        bool bad = false;
        for (int i = b + 1 + lane; i < e; i += 32)
            bad |= !(in[i].w >= in[i - 1].w);
        double dur = 0.0;
        int sg = seg_off[tr] + lane; // build id of the set
        // by the points left: the first point's number may pass 2^31 at the end
        for (int left = e - b - lane * K; left > 0; left -= 32 * K, sg += 32) {
            const int f = e - left, cnt = min(K, left);
            const float tA = in[f].w;
            dur += (double)in[f + cnt - 1].w - (double)tA;
            range[sg] = make_int4(f, cnt, tr, 0);
            keys[sg] = ((unsigned long long)f2ord(tA) << 32) | (unsigned)sg;
        }
        for (int o = 16; o > 0; o >>= 1)
            dur += __shfl_xor_sync(0xffffffffu, dur, o);
        if (__any_sync(0xffffffffu, bad) && lane == 0)
            atomicOr(meta + META_FLAG, (unsigned)BAD_ORDER);
        if (lane == 0 && dur != 0.0)
            atomicAdd((double *)(meta + META_DUR), dur);
        return;
    }
    // [0] largest |scaled coordinate|; [1 + 2 d], [2 + 2 d] axis d's minimum
    // and maximum
    __shared__ unsigned int s[VAL_THREADS / 32][9];
    unsigned int m[9] = {0u, 0xffffffffu, 0u, 0xffffffffu, 0u, 0xffffffffu, 0u, 0xffffffffu, 0u};
    bool bad = false;
    for (int64_t i = blockIdx.x * VAL_THREADS + threadIdx.x; i < n; i += pblocks * VAL_THREADS) {
        const float4 v = in[i];
        out[i] = v;
        if (fabsf(v.x) <= 1e15f && fabsf(v.y) <= 1e15f && fabsf(v.z) <= 1e15f && fabsf(v.w) <= 1e15f)
            m[0] = max(m[0], __float_as_uint(fmaxf(fmaxf(fabsf(s0 * v.x), fabsf(s1 * v.y)), fabsf(s2 * v.z))));
        else
            bad = true;
        const float c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const unsigned int u = f2ord(c[d]);
            m[1 + 2 * d] = min(m[1 + 2 * d], u);
            m[2 + 2 * d] = max(m[2 + 2 * d], u);
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0)
        atomicOr(meta + META_FLAG, (unsigned)BAD_VALUE);
#pragma unroll
    for (int d = 0; d < 9; ++d) {
        m[d] = (d & 1) ? __reduce_min_sync(0xffffffffu, m[d]) : __reduce_max_sync(0xffffffffu, m[d]);
        if (lane == 0)
            s[w][d] = m[d];
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        const int d = threadIdx.x;
        unsigned int r = s[0][d];
        for (int j = 1; j < VAL_THREADS / 32; ++j)
            r = (d & 1) ? min(r, s[j][d]) : max(r, s[j][d]);
        if (d & 1)
            atomicMin(meta + META_CMAX + d, r);
        else
            atomicMax(meta + META_CMAX + d, r);
    }
}

// AB' of one axis, sqrt(s) b - A', with its roundings spelled out: the grid
// key is taken from it twice (sort keys, extents) and both must agree, whatever
// the compiler would contract around them.
__device__ __forceinline__ float scaled_step(double q, float b, float a) { return (float)fma(q, (double)b, -(double)a); }

// One thread per segment (build order).  FP64, rounded once to the stored
// FP32 record:
//   A' = fl(sqrt(s) A),  AB' = fl(sqrt(s) B - A'),  U' = fl(AB' / |AB'|^2)
// The stored segment is [A', A' + AB'] (both exactly representable);
// r bounds, with upward rounding, the distance of every member's scaled
// position sqrt(s) p_j to it (Sec. 3.4 E_app, in the cylinder reading).
//
// FP64 instructions bound this kernel (one warp instruction occupies the pipe
// of an SM for 16 cycles).  Only the largest distance is kept, so a pass in
// FP32 first finds the members that can hold it: with offsets taken from the
// first member (small numbers) its error is below 2^-19 (|D| + |AB|)_max, and
// the members whose distance is within 2^-17 of that scale of the largest one
// are measured in FP64: one, now and then two; three or more (or a segment
// whose |AB|^2 FP32 does not hold) measure all members.  The same radius, bit
// for bit; 20,000 segments of 20 points (cold caches): 45 us with every member
// in FP64 by four lanes per segment, 23 us now.
#define SF_THREADS 128
__global__ void __launch_bounds__(SF_THREADS)
    k_segment_fit(const float4 *__restrict__ p, const int4 *__restrict__ range, int S, double q0, double q1,
                  double q2, float4 *__restrict__ rec, unsigned int *rmax_bits)
{
    const int s = blockIdx.x * SF_THREADS + threadIdx.x;
    unsigned int rbits = 0u;
    if (s < S) {
        const int4 rg = range[s];
        const int first = rg.x, count = rg.y, tr = rg.z;
        const float4 pa = p[first], pb = p[first + count - 1];
        double A[3], AB[3];
        float Af[3], ABf[3], Uf[3], res[3];
        const double qq[3] = {q0, q1, q2};
        const float qf[3] = {(float)q0, (float)q1, (float)q2};
        const float pav[3] = {pa.x, pa.y, pa.z}, pbv[3] = {pb.x, pb.y, pb.z};
        // mag only scales the rounding slack below, which is about a thousand
        // times the FP64 error of the distances; FP32 is ample for it.
        float mag = 0.f;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double sa = qq[i] * (double)pav[i];
            Af[i] = (float)sa;
            A[i] = (double)Af[i];
            res[i] = (float)(sa - A[i]); // sqrt(s) p - A' = sqrt(s) (p - p_a) + res
            ABf[i] = scaled_step(qq[i], pbv[i], Af[i]);
            AB[i] = (double)ABf[i];
            mag += fabsf(Af[i]) + fabsf((float)(A[i] + AB[i]));
        }
        const double ab2 = AB[0] * AB[0] + AB[1] * AB[1] + AB[2] * AB[2];
        // Any lam in [0, 1] names a point of the segment, so the distance to
        // it bounds the distance to the segment from above: lam = dot / |AB|^2
        // may take the reciprocal (one division, not one per member).
        const double inv_ab2 = ab2 > 0.0 ? 1.0 / ab2 : 0.0;
        // ---- FP32: squared distances, their maximum, the scale of the error
        const float ab2f = (float)ab2;
        const bool screen = ab2f > 1e-20f && ab2f < 1e35f; // else every member in FP64
        const float inv32 = (float)inv_ab2;
        auto dist2_32 = [&](const float4 &v, float &dm) {
            const float D0 = fmaf(qf[0], v.x - pa.x, res[0]), D1 = fmaf(qf[1], v.y - pa.y, res[1]),
                        D2 = fmaf(qf[2], v.z - pa.z, res[2]);
            const float lam = __saturatef(fmaf(D2, ABf[2], fmaf(D1, ABf[1], D0 * ABf[0])) * inv32);
            const float e0 = fmaf(-lam, ABf[0], D0), e1 = fmaf(-lam, ABf[1], D1), e2 = fmaf(-lam, ABf[2], D2);
            dm = fmaxf(fmaxf(fabsf(D0), fabsf(D1)), fabsf(D2));
            return fmaf(e2, e2, fmaf(e1, e1, e0 * e0));
        };
        // the three largest, and where the first two are
        float m1 = -1.f, m2 = -1.f, m3 = -1.f, dmax = 0.f;
        int j1 = 0, j2 = 0;
#pragma unroll 4
        for (int j = 0; j < count; ++j) {
            const float4 v = p[first + j];
            float dm;
            const float e = dist2_32(v, dm);
            m3 = e > m2 ? m2 : fmaxf(m3, e);
            j2 = e > m1 ? j1 : e > m2 ? j : j2;
            m2 = e > m1 ? m1 : fmaxf(m2, e);
            j1 = e > m1 ? j : j1;
            m1 = fmaxf(m1, e);
            dmax = fmaxf(dmax, dm);
            mag = fmaxf(mag, fabsf(qf[0] * v.x) + fabsf(qf[1] * v.y) + fabsf(qf[2] * v.z));
        }
        const float abm = fmaxf(fmaxf(fabsf(ABf[0]), fabsf(ABf[1])), fabsf(ABf[2]));
        const float thr = fmaxf(sqrtf(fmaxf(m1, 0.0f)) - 0x1p-17f * (dmax + abm), 0.0f);
        const float thr2 = thr * thr * (1.0f - 0x1p-20f);
        // ---- FP64: the members that can be the farthest
        auto dist2_64 = [&](int j) {
            const float4 v = p[first + j];
            const double D0 = qq[0] * (double)v.x - A[0], D1 = qq[1] * (double)v.y - A[1],
                         D2 = qq[2] * (double)v.z - A[2];
            const double lam = fmin(fmax((D0 * AB[0] + D1 * AB[1] + D2 * AB[2]) * inv_ab2, 0.0), 1.0);
            const double e0 = D0 - lam * AB[0], e1 = D1 - lam * AB[1], e2 = D2 - lam * AB[2];
            return e0 * e0 + e1 * e1 + e2 * e2;
        };
        double r2;
        if (screen && m3 < thr2) {
            r2 = dist2_64(j1);
            if (!(m2 < thr2))
                r2 = fmax(r2, dist2_64(j2));
        } else {
            r2 = 0.0;
#pragma unroll 1
            for (int j = 0; j < count; ++j)
                r2 = fmax(r2, dist2_64(j));
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
            Uf[i] = ab2 > 1e-30 ? (float)(AB[i] * inv_ab2) : 0.f;
        // FP64 rounding of the distances above is far below 1e-12 * mag.
        const double r = sqrt(r2) + 1e-12 * (1.0 + (double)mag);
        const float rf = __double2float_ru(r);
        rbits = __float_as_uint(rf); // rf >= 0: the bits order like the values
        float4 *out = rec + 4 * (size_t)s;
        out[0] = make_float4(Af[0], Af[1], Af[2], pa.w);
        out[1] = make_float4(Uf[0], Uf[1], Uf[2], pb.w);
        out[2] = make_float4(ABf[0], ABf[1], ABf[2], rf);
        out[3] = make_float4(__int_as_float(first), __int_as_float(count), __int_as_float(tr), __int_as_float(s));
    }
    rbits = __reduce_max_sync(0xffffffffu, rbits); // one atomic per warp
    if ((threadIdx.x & 31) == 0 && rbits != 0u)
        atomicMax(rmax_bits, rbits);
}

__global__ void k_time_keys(const float4 *__restrict__ p, int n,
                            unsigned long long *__restrict__ keys, int n2)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        keys[i] = ((unsigned long long)f2ord(p[i].w) << 32) | (unsigned)i;
    else if (i < n2)
        keys[i] = ~0ull;
}

// ------------------------------------------------------------ bitonic sort
//
// Batcher's bitonic network on n2 = 2^p 64-bit keys, ascending.  Step (k, j)
// compares positions i and i + j (bit j of i clear) and puts the smaller key
// first when bit k of i is clear, last otherwise.  Every kernel below keeps
// four consecutive keys per thread in registers: steps j = 1, 2 stay inside a
// thread, steps 4 <= j <= 64 inside a warp (shuffles, no barrier), steps
// 128 <= j < block size go through shared memory, and larger steps through
// distributed shared memory (cluster) or global memory.

#define BS_MIN 2048  // smallest n2 handed out (a cluster of 8 x 256 keys)
#define BS_BLOCK 4096 // keys per CTA of the multi-launch path (1024 threads)

__device__ __forceinline__ void cmpx(unsigned long long &a,
                                     unsigned long long &b, bool asc)
{
    if ((a > b) == asc) {
        unsigned long long t = a;
        a = b;
        b = t;
    }
}

__device__ __forceinline__ void bs_load4(unsigned long long (&r)[4], const unsigned long long *p)
{
    const ulonglong2 a = ((const ulonglong2 *)p)[0], b = ((const ulonglong2 *)p)[1];
    r[0] = a.x;
    r[1] = a.y;
    r[2] = b.x;
    r[3] = b.y;
}

__device__ __forceinline__ void bs_store4(unsigned long long *p, const unsigned long long (&r)[4])
{
    ((ulonglong2 *)p)[0] = make_ulonglong2(r[0], r[1]);
    ((ulonglong2 *)p)[1] = make_ulonglong2(r[2], r[3]);
}

// Steps j, j/2, ..., 1 (j <= 64) of stage k on the four keys at global
// positions g0 .. g0 + 3 (g0 a multiple of 4); the partner of a key at
// distance j >= 4 sits in lane ^ (j / 4) of the same warp.
__device__ __forceinline__ void bs_warp_steps(unsigned long long (&r)[4], int g0, int k, int j)
{
    for (; j >= 4; j >>= 1) {
        const int ld = j >> 2;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned long long w = __shfl_xor_sync(0xffffffffu, r[e], ld);
            const int g = g0 + e;
            const bool take_min = ((g & j) == 0) == ((g & k) == 0);
            const bool w_lt = w < r[e];
            r[e] = (take_min == w_lt) ? w : r[e];
        }
    }
    if (j >= 2) { // k >= 4: the four keys share bit k
        const bool asc = (g0 & k) == 0;
        cmpx(r[0], r[2], asc);
        cmpx(r[1], r[3], asc);
    }
    cmpx(r[0], r[1], (g0 & k) == 0);
    cmpx(r[2], r[3], ((g0 + 2) & k) == 0);
}

// Steps j, j/2, ..., 1 (j < nl) of stage k on a CTA's nl consecutive keys
// starting at global position gb, held four per thread (nl / 4 threads);
// s has room for nl keys.
__device__ __forceinline__ void bs_local_steps(unsigned long long (&r)[4], unsigned long long *s,
                                               int nl, int gb, int k, int j)
{
    const int t = threadIdx.x, nt = nl >> 2;
    if (j >= 128) {
        bs_store4(s + 4 * t, r);
        __syncthreads();
        for (; j >= 128; j >>= 1) {
            for (int q = t; q < (nl >> 1); q += nt) {
                const int i = ((q & ~(j - 1)) << 1) | (q & (j - 1)); // j is a power of two
                cmpx(s[i], s[i + j], ((gb + i) & k) == 0);
            }
            __syncthreads();
        }
        bs_load4(r, s + 4 * t); // each thread rereads only its own four slots
    }
    bs_warp_steps(r, gb + 4 * t, k, j);
}

// Stages 2 .. BS_BLOCK, each 4096-key block on its own (the direction of a
// block follows its global position, as the network requires).
__global__ void __launch_bounds__(BS_BLOCK / 4) k_bitonic_block(unsigned long long *keys)
{
    __shared__ __align__(16) unsigned long long s[BS_BLOCK];
    const int base = blockIdx.x * BS_BLOCK;
    unsigned long long r[4];
    bs_load4(r, keys + base + 4 * threadIdx.x);
    for (int k = 2; k <= BS_BLOCK; k <<= 1)
        bs_local_steps(r, s, BS_BLOCK, base, k, k >> 1);
    bs_store4(keys + base + 4 * threadIdx.x, r);
}

// Steps j < BS_BLOCK of stage k, inside each block.
__global__ void __launch_bounds__(BS_BLOCK / 4) k_bitonic_merge_local(unsigned long long *keys, int k)
{
    __shared__ __align__(16) unsigned long long s[BS_BLOCK];
    const int base = blockIdx.x * BS_BLOCK;
    unsigned long long r[4];
    bs_load4(r, keys + base + 4 * threadIdx.x);
    bs_local_steps(r, s, BS_BLOCK, base, k, BS_BLOCK >> 1);
    bs_store4(keys + base + 4 * threadIdx.x, r);
}

__global__ void k_bitonic_global(unsigned long long *keys, int j, int k)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x; // one per pair
    int i = ((t & ~(j - 1)) << 1) | (t & (j - 1)); // j is a power of two
    bool asc = (i & k) == 0;
    unsigned long long a = keys[i], b = keys[i + j];
    if ((a > b) == asc) {
        keys[i] = b;
        keys[i + j] = a;
    }
}

int tnn_next_pow2_sort(int64_t n)
{
    int64_t p = BS_MIN;
    while (p < n)
        p <<= 1;
    return (int)p;
}

// The whole network for n2 <= 32768 keys in one launch: a cluster of 8 CTAs
// of n2 / 32 threads, CTA c holding keys c * n2 / 8 .. (c + 1) * n2 / 8 - 1.
// A step whose partner lies in another CTA (j >= n2 / 8) publishes the keys
// in shared memory and reads the partner's through distributed shared memory
// between two cluster barriers: the first makes every key visible, the
// second keeps a CTA from overwriting (or leaving) its buffer while its
// partner still reads it.
#define BS_CLUSTER 8
#define BS_CLUSTER_MAX (BS_CLUSTER * 4096)

__global__ void __cluster_dims__(BS_CLUSTER, 1, 1) __launch_bounds__(1024)
    k_bitonic_cluster(unsigned long long *keys, int n2)
{
    __shared__ __align__(16) unsigned long long s[4096];
    cg::cluster_group cluster = cg::this_cluster();
    const int c = (int)cluster.block_rank(), nl = n2 / BS_CLUSTER, base = c * nl;
    const int g0 = base + 4 * threadIdx.x;
    unsigned long long r[4];
    bs_load4(r, keys + g0);
    for (int k = 2; k <= n2; k <<= 1) {
        int j = k >> 1;
        for (; j >= nl; j >>= 1) {
            const unsigned long long *peer = cluster.map_shared_rank(s, c ^ (j / nl));
            bs_store4(s + 4 * threadIdx.x, r);
            cluster.sync();
            unsigned long long w[4];
            bs_load4(w, peer + 4 * threadIdx.x);
            const bool take_min = ((g0 & j) == 0) == ((g0 & k) == 0); // same for g0 .. g0 + 3
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool w_lt = w[e] < r[e];
                r[e] = (take_min == w_lt) ? w[e] : r[e];
            }
            cluster.sync();
        }
        bs_local_steps(r, s, nl, base, k, j);
    }
    bs_store4(keys + g0, r);
}

void tnn_bitonic_sort(unsigned long long *keys, int n2, cudaStream_t st)
{
    if (n2 <= BS_CLUSTER_MAX) {
        k_bitonic_cluster<<<BS_CLUSTER, n2 / (4 * BS_CLUSTER), 0, st>>>(keys, n2);
        return;
    }
    k_bitonic_block<<<n2 / BS_BLOCK, BS_BLOCK / 4, 0, st>>>(keys);
    for (int64_t k = 2 * BS_BLOCK; k <= n2; k <<= 1) { // n2 is at most 2^30
        for (int j = (int)(k >> 1); j >= BS_BLOCK; j >>= 1)
            k_bitonic_global<<<(n2 / 2 + 255) / 256, 256, 0, st>>>(keys, j, (int)k);
        k_bitonic_merge_local<<<n2 / BS_BLOCK, BS_BLOCK / 4, 0, st>>>(keys, (int)k);
    }
}

// -------------------------------------------------------------- radix sort
//
// Stable ascending sort by the upper halves of n2 <= 32,768 keys in one
// launch, least significant 8 bits first: a cluster of 8 CTAs, CTA c holding
// positions c nl .. (c + 1) nl - 1 (nl = n2 / 8), IT keys per thread.  Per
// digit: ranks inside a warp by match, per-warp counts in shared memory, their
// prefix over the warps, the CTAs' totals exchanged through distributed shared
// memory, and every key written straight into its place in the CTA that holds
// it.  Keys carry their position below the sort value, so a stable sort by the
// value is the sort of the whole key.  Latency bounds it: two cluster barriers
// per digit (four digits for times, as many as the number of grid keys needs)
// against two per step of the bitonic network whose partner is in another CTA;
// 20,000 keys (cold caches): 46 us by the network, 25 us for times and 14 us
// for grid keys.
#define RS_CLUSTER 8

struct RadixSmem {
    unsigned long long buf[4096];
    unsigned short hist[32][256]; // per warp: count, then prefix over the warps
    unsigned tot[256];            // this CTA's count per digit (read by its peers)
    unsigned off[256];            // first position of this CTA's keys per digit
    unsigned part[8];
};

template <int IT>
__global__ void __cluster_dims__(RS_CLUSTER, 1, 1) __launch_bounds__(1024)
    k_radix_cluster(unsigned long long *keys, int n2, int bits)
{
    extern __shared__ __align__(16) unsigned char raw[];
    RadixSmem &S = *(RadixSmem *)raw;
    cg::cluster_group cluster = cg::this_cluster();
    const int c = (int)cluster.block_rank(), nl = n2 / RS_CLUSTER, t = threadIdx.x;
    const int lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    const int at = w * 32 * IT + lane; // key j of this thread: position at + 32 j of the CTA
    unsigned long long r[IT];
#pragma unroll
    for (int j = 0; j < IT; ++j)
        r[j] = keys[(size_t)c * nl + at + 32 * j];
#pragma unroll 1
    for (int shift = 32; shift < 32 + bits; shift += 8) {
        for (int i = t; i < nw * 256; i += blockDim.x)
            (&S.hist[0][0])[i] = 0;
        __syncthreads();
        int rank[IT];
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            const unsigned d = (unsigned)(r[j] >> shift) & 255u;
            const unsigned same = __match_any_sync(0xffffffffu, d);
            const unsigned before = same & ((1u << lane) - 1u);
            rank[j] = S.hist[w][d] + __popc(before);
            __syncwarp();
            if (before == 0)
                S.hist[w][d] = (unsigned short)(S.hist[w][d] + __popc(same));
            __syncwarp();
        }
        __syncthreads();
        if (t < 256) {
            unsigned sum = 0;
#pragma unroll 8
            for (int i = 0; i < nw; ++i) {
                const unsigned h = S.hist[i][t];
                S.hist[i][t] = (unsigned short)sum;
                sum += h;
            }
            S.tot[t] = sum;
        }
        // every key of this digit is in registers, every total is visible
        cluster.sync();
        unsigned all = 0, mine = 0;
        if (t < 256) {
#pragma unroll
            for (int i = 0; i < RS_CLUSTER; ++i) {
                const unsigned v = *cluster.map_shared_rank(&S.tot[t], i);
                all += v;
                mine += i < c ? v : 0u;
            }
            unsigned inc = all;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o)
                    inc += v;
            }
            if (lane == 31)
                S.part[w] = inc;
            mine += inc - all;
        }
        __syncthreads();
        if (t < 256) {
            for (int i = 0; i < w; ++i)
                mine += S.part[i];
            S.off[t] = mine;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            const unsigned d = (unsigned)(r[j] >> shift) & 255u;
            const unsigned pos = S.off[d] + S.hist[w][d] + (unsigned)rank[j];
            const unsigned dst = pos / (unsigned)nl;
            *cluster.map_shared_rank(&S.buf[pos - dst * (unsigned)nl], dst) = r[j];
        }
        cluster.sync(); // every key is in place
#pragma unroll
        for (int j = 0; j < IT; ++j)
            r[j] = S.buf[at + 32 * j];
    }
#pragma unroll
    for (int j = 0; j < IT; ++j)
        keys[(size_t)c * nl + at + 32 * j] = r[j];
}

// Ascending sort of n2 keys (sort value << 32 | position, in the order of
// their positions, padding ~0 behind them); the values fit in `bits` bits and
// are not all ones there.
static tnn_status sort_by_value(unsigned long long *keys, int n2, int bits, cudaStream_t st)
{
    if (n2 > RS_CLUSTER * 4096) {
        tnn_bitonic_sort(keys, n2, st);
        return TNN_OK;
    }
    const int nl = n2 / RS_CLUSTER, threads = std::min(nl, 1024), it = nl / threads;
    const auto kern = it == 1 ? k_radix_cluster<1> : it == 2 ? k_radix_cluster<2> : k_radix_cluster<4>;
    TNN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixSmem)));
    kern<<<RS_CLUSTER, threads, sizeof(RadixSmem), st>>>(keys, n2, bits);
    TNN_CUDA_TRY(cudaGetLastError());
    return TNN_OK;
}

// --------------------------------------------------------- gather / scans

// Running maximum of t_B over the t_A order, in two passes over blocks of
// 1024 segments: the maximum of every block, then per block the maxima of
// the blocks before it and a block-wide inclusive scan.
__device__ __forceinline__ float block_max_1024(float v, float *sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0)
        sh[w] = v;
    __syncthreads();
    v = sh[lane];
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    return v;
}

// The records in t_A order (keys hold build ids), their start times, the
// position of every build id, and the block maxima.
__global__ void __launch_bounds__(1024)
    k_gather_segments(const unsigned long long *__restrict__ keys, const float4 *__restrict__ rec, int S,
                      float4 *__restrict__ out, float *__restrict__ tA, int32_t *__restrict__ pos,
                      float *__restrict__ bmax)
{
    __shared__ float sh[32];
    const int i = blockIdx.x * 1024 + threadIdx.x;
    float tB = -INFINITY;
    if (i < S) {
        const int s = (int)(keys[i] & 0xffffffffu);
        pos[s] = i;
        const float4 *r = rec + 4 * (size_t)s;
        float4 *o = out + 4 * (size_t)i;
        const float4 a = r[0], u = r[1];
        o[0] = a;
        o[1] = u;
        o[2] = r[2];
        o[3] = r[3];
        tA[i] = a.w;
        tB = u.w;
    }
    const float v = block_max_1024(tB, sh);
    if (threadIdx.x == 0)
        bmax[blockIdx.x] = v;
}

__global__ void __launch_bounds__(1024) k_pm_apply(const float4 *__restrict__ seg, int S,
                                                   const float *__restrict__ bmax,
                                                   float *__restrict__ pm)
{
    __shared__ float sh[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float c = -INFINITY;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += 1024)
        c = fmaxf(c, bmax[b]);
    const float carry = block_max_1024(c, sh);
    const int i = blockIdx.x * 1024 + threadIdx.x;
    float v = i < S ? seg[4 * (size_t)i + 1].w : -INFINITY;
    for (int o = 1; o < 32; o <<= 1) {
        const float u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o)
            v = fmaxf(v, u);
    }
    if (lane == 31)
        sh[w] = v;
    __syncthreads();
    if (w == 0) {
        float y = sh[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const float u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o)
                y = fmaxf(y, u);
        }
        sh[lane] = y;
    }
    __syncthreads();
    if (w > 0)
        v = fmaxf(v, sh[w - 1]);
    if (i < S)
        pm[i] = fmaxf(v, carry);
}

__global__ void k_gather_points(const unsigned long long *__restrict__ keys,
                                const float4 *__restrict__ p, int n,
                                float4 *__restrict__ out,
                                int32_t *__restrict__ idx)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    int j = (int)(keys[i] & 0xffffffffu);
    out[i] = p[j];
    idx[i] = j;
}

// ------------------------------------------------------------------- grid

__device__ __forceinline__ float ord2f(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

struct GridBuild {
    float x0, y0, cell, inv_cell, t0, dt, inv_dt;
    int nx, ny, ncell, nb;
};

// Grid key of a segment: bucket of t_A, cell of the midpoint of [A', A' + AB'].
__device__ __forceinline__ int grid_key(const GridBuild &g, float tA, float ax, float ay, float bx, float by,
                                        int &bk, int &cx, int &cy)
{
    const float mx = fmaf(0.5f, bx, ax), my = fmaf(0.5f, by, ay);
    bk = min(max((int)floorf((tA - g.t0) * g.inv_dt), 0), g.nb - 1);
    cx = min(max((int)floorf((mx - g.x0) * g.inv_cell), 0), g.nx - 1);
    cy = min(max((int)floorf((my - g.y0) * g.inv_cell), 0), g.ny - 1);
    return bk * g.ncell + cy * g.nx + cx;
}

// Sort keys (grid key << 32 | build id) straight from the end points, with
// the segment fit's rounding: they need none of its radii, so their sort runs
// beside the fit.
__global__ void k_grid_sort_keys(const float4 *__restrict__ p, const int4 *__restrict__ range, int S, int S2,
                                 double q0, double q1, const __grid_constant__ GridBuild g,
                                 unsigned long long *__restrict__ keys)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x; // build id
    if (s >= S) {
        if (s < S2)
            keys[s] = ~0ull; // the sort's padding
        return;
    }
    const int4 r = range[s];
    const float4 pa = p[r.x], pb = p[r.x + r.y - 1];
    const float ax = (float)(q0 * (double)pa.x), ay = (float)(q1 * (double)pa.y);
    const float bx = scaled_step(q0, pb.x, ax), by = scaled_step(q1, pb.y, ay);
    int bk, cx, cy;
    const int key = grid_key(g, pa.w, ax, ay, bx, by, bk, cx, cy);
    keys[s] = ((unsigned long long)(unsigned)key << 32) | (unsigned)s;
}

// The per-key aggregates of the records: the extent (FP64, rounded up) of the
// member cylinders around the key's cell rectangle and the largest t_B; the
// per-bucket largest t_B.
__global__ void k_grid_extents(const float4 *__restrict__ seg, int S, const __grid_constant__ GridBuild g,
                               unsigned int *__restrict__ ext_bits, unsigned int *__restrict__ tB_ord,
                               unsigned int *__restrict__ bmax_ord)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x; // build id
    if (p >= S)
        return;
    const float4 *r = seg + 4 * (size_t)p;
    const float4 a = r[0], u = r[1], b = r[2];
    int bk, cx, cy;
    const int key = grid_key(g, a.w, a.x, a.y, b.x, b.y, bk, cx, cy);
    // every cylinder point is within |AB|/2 + r of the midpoint
    const double ax = a.x, ay = a.y, bx = b.x, by = b.y, bz = b.z;
    const double half = 0.5 * sqrt(bx * bx + by * by + bz * bz) + (double)b.w;
    const double Mx = ax + 0.5 * bx, My = ay + 0.5 * by;
    const double rx0 = (double)g.x0 + cx * (double)g.cell, rx1 = rx0 + g.cell;
    const double ry0 = (double)g.y0 + cy * (double)g.cell, ry1 = ry0 + g.cell;
    const double dx = fmax(fmax(rx0 - Mx, Mx - rx1), 0.0);
    const double dy = fmax(fmax(ry0 - My, My - ry1), 0.0);
    // margin for the FP32 evaluation of the rectangle corners at query time
    const double margin = 1e-6 * (fabs((double)g.x0) + fabs((double)g.y0) +
                                  (double)g.cell * (g.nx + g.ny + 2)) + 1e-9;
    const float e = __double2float_ru(sqrt(dx * dx + dy * dy) + half + margin);
    atomicMax(ext_bits + key, __float_as_uint(e));
    atomicMax(tB_ord + key, f2ord(u.w));
    atomicMax(bmax_ord + bk, f2ord(u.w));
}

struct GridTail {
    const unsigned long long *keys; // sorted (grid key << 32 | build id)
    const float4 *rec;              // build order
    const int32_t *pos;             // t_A position of every build id
    int S, nkeys, nb, kblocks, rblocks;
    int32_t *off, *ids;
    float4 *gseg;
    float *ext, *tB, *bpm;
    int4 *krec;
    unsigned int *ext_max;
};

#define GT_THREADS 256
#define GT_STAGE 2048

// Everything the grid needs from its sorted keys, by block:
//   the first kblocks   256 keys each: CSR offsets (the block's slice of the
//                       sorted keys is found once and searched in shared
//                       memory), largest t_B decoded, the 16-byte key record,
//                       the largest extent;
//   the next rblocks    segment records in key order (record 3's trajectory
//                       field replaced by the t_A position), so that the
//                       search reads a key's segments without an indirection;
//   the last one        running maximum of t_B over the buckets.
// (Eight kernels before, four of them a search of all keys or less than one
// wave of work each, 33 us one after the other at 20,000 segments; 5 us.)
__global__ void __launch_bounds__(GT_THREADS) k_grid_tail(const __grid_constant__ GridTail g)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int b = blockIdx.x;
    if (b < g.kblocks) {
        __shared__ int s_lo[2], s_off[GT_THREADS + 1];
        __shared__ unsigned s_key[GT_STAGE];
        const int k0 = b * GT_THREADS;
        // segments of keys [k0, k0 + 256): a 32-way search of one warp each
        if (w < 2) {
            const unsigned kt = (unsigned)(k0 + w * GT_THREADS);
            int lo = 0, hi = g.S; // every index < lo is below, every index >= hi is not
            while (hi > lo) {
                const int step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step - 1;
                const bool lt = at < hi && (unsigned)(g.keys[at] >> 32) < kt;
                const int n = __popc(__ballot_sync(0xffffffffu, lt));
                const int nlo = min(lo + n * step, hi);
                hi = min(hi, lo + (n + 1) * step - 1);
                lo = nlo;
            }
            if (lane == 0)
                s_lo[w] = lo;
        }
        __syncthreads();
        const int lo = s_lo[0], m = s_lo[1] - lo;
        const bool staged = m <= GT_STAGE;
        if (staged)
            for (int i = t; i < m; i += GT_THREADS)
                s_key[i] = (unsigned)(g.keys[lo + i] >> 32);
        __syncthreads();
        const int k = k0 + t;
        {
            int l = 0, h = m; // first of the slice not below k
            while (l < h) {
                const int mid = (l + h) >> 1;
                const unsigned v = staged ? s_key[mid] : (unsigned)(g.keys[lo + mid] >> 32);
                if (v < (unsigned)k)
                    l = mid + 1;
                else
                    h = mid;
            }
            s_off[t] = lo + l;
        }
        if (t == 0)
            s_off[GT_THREADS] = lo + m;
        __syncthreads();
        unsigned int e = 0;
        if (k < g.nkeys) {
            const int o0 = s_off[t], o1 = s_off[t + 1];
            e = __float_as_uint(g.ext[k]); // extents are non-negative: the bits order them
            const unsigned int u = __float_as_uint(g.tB[k]);
            const float tB = u ? ord2f(u) : -INFINITY;
            g.tB[k] = tB;
            g.off[k] = o0;
            g.krec[k] = make_int4(o0, o1, (int)e, __float_as_int(tB));
            if (k == g.nkeys - 1)
                g.off[g.nkeys] = o1;
        }
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0 && e)
            atomicMax(g.ext_max, e);
        return;
    }
    b -= g.kblocks;
    if (b < g.rblocks) {
        const int i = b * GT_THREADS + t;
        if (i >= g.S)
            return;
        const int s = (int)(g.keys[i] & 0xffffffffu), p = g.pos[s];
        g.ids[i] = p;
        g.gseg[4 * (size_t)i] = g.rec[4 * (size_t)s];
        g.gseg[4 * (size_t)i + 1] = g.rec[4 * (size_t)s + 1];
        g.gseg[4 * (size_t)i + 2] = g.rec[4 * (size_t)s + 2];
        float4 r3 = g.rec[4 * (size_t)s + 3];
        r3.z = __int_as_float(p);
        g.gseg[4 * (size_t)i + 3] = r3;
        return;
    }
    // buckets: 256 per step, the running maximum carried over
    __shared__ float s_w[GT_THREADS / 32];
    float carry = -INFINITY;
    for (int i0 = 0; i0 < g.nb; i0 += GT_THREADS) {
        const int i = i0 + t;
        const unsigned int u = i < g.nb ? __float_as_uint(g.bpm[i]) : 0u;
        float v = u ? ord2f(u) : -INFINITY;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float x = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o)
                v = fmaxf(v, x);
        }
        if (lane == 31)
            s_w[w] = v;
        __syncthreads();
        float all = carry;
        for (int j = 0; j < GT_THREADS / 32; ++j) {
            if (j == w)
                v = fmaxf(v, all); // the warps and steps before
            all = fmaxf(all, s_w[j]);
        }
        if (i < g.nb)
            g.bpm[i] = v;
        carry = all;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- host API

// The index may still be read by work queued on any stream: wait for the
// device (as cudaFree would), then return the arrays to the pool.
// Arrays back to the pool in the order of `st`, host parts freed.
static void release_index(tnn_index *ix, cudaStream_t st)
{
    void *arrays[] = {ix->mem_seg, ix->mem_grid, ix->pts_t, ix->idx_t, ix->pts_k,
                      ix->idx_k,   ix->kp_start, ix->pts_m, ix->idx_m, ix->code_m};
    for (void *p : arrays)
        tnn_free(p, st);
    free(ix->h_tiles);
    if (ix->built)
        cudaEventDestroy(ix->built);
    delete ix;
}

static void free_index(tnn_index *ix)
{
    if (!ix)
        return;
    cudaDeviceSynchronize();
    release_index(ix, 0);
}

void tnn_index_release(tnn_index *ix, cudaStream_t st)
{
    if (ix)
        release_index(ix, st);
}

// The build's two further streams per device (non-blocking, created on first
// use): the t_A sort and the grid-key sort run there beside the segment fit.
#define TNN_BUILD_MAX_DEVICES 64
static std::mutex g_side_mu;
static cudaStream_t g_side_stream[TNN_BUILD_MAX_DEVICES][2];

static cudaError_t side_streams(int dev, cudaStream_t out[2])
{
    if (dev < 0 || dev >= TNN_BUILD_MAX_DEVICES)
        return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_side_mu);
    for (int i = 0; i < 2; ++i) {
        if (!g_side_stream[dev][i]) {
            cudaError_t e = cudaStreamCreateWithFlags(&g_side_stream[dev][i], cudaStreamNonBlocking);
            if (e != cudaSuccess)
                return e;
        }
        out[i] = g_side_stream[dev][i];
    }
    return cudaSuccess;
}

// Events of this host thread on one device, kept between builds: after the
// validation, its read-back, the t_A sort, the grid keys, the segment fit.
struct BuildEvents {
    cudaEvent_t e[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    ~BuildEvents()
    {
        for (cudaEvent_t x : e)
            if (x)
                cudaEventDestroy(x);
    }
    cudaError_t get()
    {
        for (cudaEvent_t &x : e)
            if (!x) {
                const cudaError_t r = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
                if (r != cudaSuccess) {
                    x = nullptr;
                    return r;
                }
            }
        return cudaSuccess;
    }
};

// Build-time scratch, returned to the pool in stream order.
struct DevBuf {
    void *p = nullptr;
    cudaStream_t st = 0;
    cudaError_t alloc(size_t bytes, cudaStream_t s)
    {
        st = s;
        return tnn_alloc(&p, bytes, s);
    }
    ~DevBuf() { tnn_free(p, st); }
};

// Consecutive arrays of one allocation, each on a 256-byte boundary: sized
// first (base NULL), then placed.
struct Carve {
    char *base;
    size_t used = 0;
    explicit Carve(void *b) : base((char *)b) {}
    template <typename T> void take(T *&p, size_t count)
    {
        if (base)
            p = (T *)(base + used);
        used += (count * sizeof(T) + 255) & ~(size_t)255;
    }
};

// Page-locked staging of this host thread for the build's uploads and the
// values it reads back (larger uploads go through pageable memory).
struct Staging {
    static constexpr size_t bytes = 1 << 20;
    unsigned char *p = nullptr;
    ~Staging()
    {
        if (p)
            cudaFreeHost(p);
    }
    cudaError_t get(unsigned char **out)
    {
        if (!p) {
            cudaError_t e = cudaHostAlloc((void **)&p, bytes, cudaHostAllocPortable);
            if (e != cudaSuccess) {
                p = nullptr;
                return e;
            }
        }
        *out = p;
        return cudaSuccess;
    }
};

static float host_ord2f(uint32_t u)
{
    uint32_t v = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    float f;
    memcpy(&f, &v, sizeof(f));
    return f;
}

// Grid geometry from the points' bounding box in sqrt(sigma)-scaled x, y
// (it holds every segment midpoint up to rounding, and keys are clamped to
// the grid), their time range and the summed segment duration.  Buckets span
// about five mean segment durations (at most 4096 of them); cells are square,
// 0.8 of them per segment of a bucket on average, at most 65,536 cells and
// 2^22 keys.  (Tile + per-query kernels, us, at 1.0 / 0.8 / 0.7 cells per
// segment: 400,000 flight samples 277 / 277 / 280, 1 M random walks 540 / 531
// / 542, 4 M samples 3,020 / 2,878 / 2,827, a half-hour-lag nowcast of 185,376
// 412 / 361 / 340; 2 cells defer more queries than they save: 4 M 4,300.)
#ifndef TNN_BUCKET_SEGS
#define TNN_BUCKET_SEGS 5.0 // bucket span in mean segment durations
#endif
#ifndef TNN_KEY_SEGS
#define TNN_KEY_SEGS 0.8 // cells per mean segment of a bucket
#endif
static GridBuild grid_geometry(double xmn, double xmx, double ymn, double ymx, double tmn,
                               double tmx, double dur, int64_t S)
{
    const double T = tmx - tmn;
    double dt = TNN_BUCKET_SEGS * dur / S;
    if (!(dt > 0.0))
        dt = T > 0.0 ? T / 64.0 : 1.0;
    if (T / dt > 4095.0)
        dt = T / 4095.0;
    const int nb = (int)std::min(4096.0, floor(T / dt) + 1.0);
    const double Wd = xmx - xmn, Hd = ymx - ymn;
    const double target = std::min(65536.0, std::max(1.0, TNN_KEY_SEGS * S / nb));
    double cell = sqrt(std::max(Wd * Hd, 1e-12) / target);
    cell = std::max(cell, std::max(std::max(Wd, Hd) / 1024.0, 1e-6));
    int nx = 1, ny = 1;
    for (;;) {
        nx = (int)floor(Wd / cell) + 1;
        ny = (int)floor(Hd / cell) + 1;
        if ((double)nx * ny <= 65536.0 && (double)nb * nx * ny <= (double)(1 << 22))
            break;
        cell *= 1.25;
    }
    GridBuild g;
    g.x0 = (float)xmn;
    g.y0 = (float)ymn;
    g.cell = (float)cell;
    g.inv_cell = (float)(1.0 / cell);
    g.t0 = (float)tmn;
    g.dt = (float)dt;
    g.inv_dt = (float)(1.0 / dt);
    g.nx = nx;
    g.ny = ny;
    g.ncell = nx * ny;
    g.nb = nb;
    return g;
}

// The grid's arrays, zeroed where the key kernel takes maxima.
static tnn_status grid_alloc(tnn_index *ix, const GridBuild &g, cudaStream_t st)
{
    const size_t S = (size_t)ix->S, nb = (size_t)g.nb, nkeys = nb * g.ncell;
    size_t zeroed = 0;
    for (int pass = 0; pass < 2; ++pass) {
        Carve c(ix->mem_grid);
        c.take(ix->g_ext, nkeys);
        c.take(ix->g_tB, nkeys);
        c.take(ix->g_bpm, nb);
        zeroed = c.used;
        c.take(ix->g_off, nkeys + 1);
        c.take(ix->g_ids, S);
        c.take(ix->g_seg, 4 * S);
        c.take(ix->g_krec, nkeys);
        if (pass == 0)
            TNN_CUDA_TRY(tnn_alloc(&ix->mem_grid, c.used, st));
    }
    TNN_CUDA_TRY(cudaMemsetAsync(ix->mem_grid, 0, zeroed, st));
    return TNN_OK;
}

// The grid from its sorted keys (build ids; pos = t_A position of each).
static tnn_status build_grid(tnn_index *ix, const unsigned long long *keys, const float4 *rec,
                             const int32_t *pos, const GridBuild &g, cudaStream_t st)
{
    GridTail a;
    a.keys = keys;
    a.rec = rec;
    a.pos = pos;
    a.S = (int)ix->S;
    a.nb = g.nb;
    a.nkeys = g.nb * g.ncell;
    a.kblocks = (a.nkeys + GT_THREADS - 1) / GT_THREADS;
    a.rblocks = (a.S + GT_THREADS - 1) / GT_THREADS;
    a.off = ix->g_off;
    a.ids = ix->g_ids;
    a.gseg = ix->g_seg;
    a.ext = ix->g_ext;
    a.tB = ix->g_tB;
    a.bpm = ix->g_bpm;
    a.krec = ix->g_krec;
    a.ext_max = (unsigned int *)ix->g_ext_max;
    k_grid_tail<<<a.kblocks + a.rblocks + 1, GT_THREADS, 0, st>>>(a);
    TNN_CUDA_TRY(cudaGetLastError());
    GridDesc &G = ix->grid;
    G.x0 = g.x0;
    G.y0 = g.y0;
    G.cell = g.cell;
    G.inv_cell = g.inv_cell;
    G.t0 = g.t0;
    G.dt = g.dt;
    G.inv_dt = g.inv_dt;
    G.ext_max = ix->g_ext_max;
    G.nx = g.nx;
    G.ny = g.ny;
    G.ncell = g.ncell;
    G.nb = g.nb;
    G.off = ix->g_off;
    G.ids = ix->g_ids;
    G.gseg = ix->g_seg;
    G.ext = ix->g_ext;
    G.tB = ix->g_tB;
    G.bpm = ix->g_bpm;
    G.krec = ix->g_krec;
    return TNN_OK;
}

extern "C" tnn_status tnn_build_segments(const float *d_xyzt, int64_t n,
                                         const int64_t *h_traj_off,
                                         int64_t n_traj,
                                         const tnn_build_params *params,
                                         tnn_stream_t stream, tnn_index **out)
{
    tnn_clear_error();
    TNN_ARG_CHECK(out != nullptr, "out is NULL");
    *out = nullptr;
    TNN_ARG_CHECK(params != nullptr, "params is NULL");
    TNN_ARG_CHECK(n >= 1 && n < (1ll << 31) - 64, "n must be in [1, 2^31-64), got %lld",
                  (long long)n);
    TNN_ARG_CHECK(d_xyzt != nullptr && h_traj_off != nullptr, "NULL input");
    TNN_ARG_CHECK(((uintptr_t)d_xyzt & 15) == 0, "d_xyzt must be 16-byte aligned");
    TNN_ARG_CHECK(n_traj >= 1 && n_traj <= n, "n_traj must be in [1, n]");
    const int K = params->seg_len;
    TNN_ARG_CHECK(K >= 2 && K <= 64, "seg_len must be in [2, 64], got %d", K);
    for (int i = 0; i < 4; ++i) {
        double s = params->sigma[i];
        TNN_ARG_CHECK(isfinite(s) && s >= 0.0 && s <= 1e6,
                      "sigma[%d] must be finite in [0, 1e6]", i);
    }
    TNN_ARG_CHECK(h_traj_off[0] == 0 && h_traj_off[n_traj] == n,
                  "traj_off must start at 0 and end at n");
    int64_t S = 0, nt = 0; // segments; query tiles of up to 32 points of one trajectory
    for (int64_t t = 0; t < n_traj; ++t) {
        const int64_t len = h_traj_off[t + 1] - h_traj_off[t];
        TNN_ARG_CHECK(len >= 0, "traj_off must be non-decreasing");
        S += (uint32_t)(len + K - 1) / (uint32_t)K; // len < 2^31
        nt += (len + 31) >> 5;
    }
    // the sorts take a power of two of keys in 32-bit places
    if (S > (1ll << 30)) {
        tnn_set_error("index allocation failed: %lld segments, at most 2^30 are possible", (long long)S);
        return TNN_ERR_OOM;
    }
    cudaStream_t st = (cudaStream_t)stream;

    tnn_index *ix = new tnn_index();
    memset(ix, 0, sizeof(*ix));
    cudaGetDevice(&ix->device);
    ix->n = n;
    ix->n_traj = n_traj;
    ix->S = S;
    ix->K = K;
    ix->n_tiles = nt;
    for (int i = 0; i < 4; ++i) {
        ix->sigma[i] = params->sigma[i];
        ix->sig_f[i] = (float)params->sigma[i];
    }
    for (int i = 0; i < 3; ++i)
        ix->ssq_f[i] = (float)sqrt(params->sigma[i]);

    // What goes up in one copy: the header, trajectory and segment offsets
    // per trajectory, tile starts.
    const size_t up_words = META_WORDS + 2 * (size_t)(n_traj + 1) + (size_t)(nt + 1);
    static thread_local Staging t_stage;
    unsigned char *stage = nullptr;
    std::vector<unsigned int> big;
    cudaError_t e = t_stage.get(&stage);
    unsigned int *up = (unsigned int *)stage;
    if (e == cudaSuccess && up_words * 4 > Staging::bytes - 64) {
        big.resize(up_words);
        up = big.data();
    }
    ix->h_tiles = (int32_t *)malloc(sizeof(int32_t) * (size_t)(nt + 1));
    if (e != cudaSuccess || !ix->h_tiles) {
        free_index(ix);
        tnn_set_error("index allocation failed (host tables)");
        return TNN_ERR_OOM;
    }
    int32_t *toff_h = (int32_t *)(up + META_WORDS), *soff_h = toff_h + n_traj + 1;
    {
        static const unsigned int meta_init[META_WORDS] = {0u, 0u, 0xffffffffu, 0u, 0xffffffffu, 0u,
                                                           0xffffffffu, 0u, 0xffffffffu, 0u};
        memcpy(up, meta_init, sizeof(meta_init));
        int64_t j = 0, sj = 0;
        for (int64_t t = 0; t < n_traj; ++t) {
            const int64_t a = h_traj_off[t], b = h_traj_off[t + 1];
            toff_h[t] = (int32_t)a;
            soff_h[t] = (int32_t)sj;
            sj += (uint32_t)(b - a + K - 1) / (uint32_t)K;
            for (int64_t r = a; r < b; r += 32)
                ix->h_tiles[j++] = (int32_t)r;
        }
        toff_h[n_traj] = (int32_t)n;
        soff_h[n_traj] = (int32_t)S;
        ix->h_tiles[nt] = (int32_t)n;
        memcpy(soff_h + n_traj + 1, ix->h_tiles, sizeof(int32_t) * (size_t)(nt + 1));
    }

    // One allocation for what stays before the grid's geometry is known, one
    // for the build's scratch.
    const int s2 = tnn_next_pow2_sort(S), nblk = (int)((S + 1023) / 1024);
    DevBuf scratch;
    unsigned int *d_up = nullptr;
    float4 *rec = nullptr;
    unsigned long long *keys = nullptr, *keys2 = nullptr;
    int32_t *pos = nullptr;
    float *bmax = nullptr;
    int4 *range = nullptr;
    for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {
        Carve c(ix->mem_seg), x(scratch.p);
        c.take(ix->pts, (size_t)n);
        c.take(ix->seg, 4 * (size_t)S);
        c.take(ix->segTA, (size_t)S);
        c.take(ix->segPM, (size_t)S);
        c.take(d_up, up_words);
        x.take(rec, 4 * (size_t)S);
        x.take(keys, (size_t)s2);
        x.take(keys2, (size_t)s2);
        x.take(pos, (size_t)S);
        x.take(bmax, (size_t)nblk);
        x.take(range, (size_t)S);
        if (pass == 0) {
            e = tnn_alloc(&ix->mem_seg, c.used, st);
            if (e == cudaSuccess)
                e = scratch.alloc(x.used, st);
        }
    }
    if (e != cudaSuccess) {
        free_index(ix);
        tnn_set_error("index allocation failed: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? TNN_ERR_OOM : TNN_ERR_CUDA;
    }
    unsigned int *meta = d_up;
    const int32_t *toff = (const int32_t *)(d_up + META_WORDS), *soff = toff + n_traj + 1;
    ix->d_tiles = (int32_t *)(soff + n_traj + 1);
    ix->d_rmax = meta + META_RMAX;
    ix->g_ext_max = (float *)(meta + META_EXT);
    const int tb = 256;
    static thread_local BuildEvents t_events[TNN_BUILD_MAX_DEVICES];
    cudaStream_t side[2] = {nullptr, nullptr};
    e = side_streams(ix->device, side);
    BuildEvents &ev = t_events[e == cudaSuccess ? ix->device : 0];
    if (e == cudaSuccess)
        e = ev.get();
    if (e == cudaSuccess)
        e = cudaEventCreateWithFlags(&ix->built, cudaEventDisableTiming);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_up, up, up_words * 4, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) {
        free_index(ix);
        tnn_set_error("index upload failed: %s", cudaGetErrorString(e));
        return TNN_ERR_CUDA;
    }
    const int ni = (int)n, Si = (int)S, Ti = (int)n_traj;
    // ---- validation, and what the grid geometry needs.  The values come
    // back through page-locked memory and an event, the build's only host
    // synchronisation; the t_A sort (on the first side stream) and the
    // segment fit need neither the geometry nor the validation result and run
    // while the host waits, chooses the geometry and enqueues the rest.
    // Invalid input is still reported here; their output is then dropped.
    const int pblocks = (int)std::min<int64_t>((n + 4 * VAL_THREADS - 1) / (4 * VAL_THREADS), 608);
    k_validate<<<pblocks + (Ti + VAL_THREADS / 32 - 1) / (VAL_THREADS / 32), VAL_THREADS, 0, st>>>(
        (const float4 *)d_xyzt, ix->pts, ni, ix->ssq_f[0], ix->ssq_f[1], ix->ssq_f[2], toff, soff, Ti, K, pblocks,
        Si, s2, range, keys, meta);
    unsigned int hm[META_READ], *back = (unsigned int *)(stage + Staging::bytes - 64);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaEventRecord(ev.e[0], st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(back, meta, sizeof(hm), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
        e = cudaEventRecord(ev.e[1], st);
    if (e == cudaSuccess)
        e = cudaStreamWaitEvent(side[0], ev.e[0], 0);
    const double q0 = sqrt(params->sigma[0]), q1 = sqrt(params->sigma[1]);
    if (e == cudaSuccess) {
        if (sort_by_value(keys, s2, 32, side[0]) != TNN_OK)
            e = cudaErrorUnknown;
        else
            e = cudaEventRecord(ev.e[2], side[0]);
    }
    if (e == cudaSuccess) {
        k_segment_fit<<<(Si + SF_THREADS - 1) / SF_THREADS, SF_THREADS, 0, st>>>(
            ix->pts, range, Si, q0, q1, sqrt(params->sigma[2]), rec, ix->d_rmax);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaEventSynchronize(ev.e[1]);
    if (e != cudaSuccess) {
        free_index(ix);
        tnn_set_error("index validation failed: %s", cudaGetErrorString(e));
        return TNN_ERR_CUDA;
    }
    memcpy(hm, back, sizeof(hm));
    if (hm[META_FLAG] & BAD_VALUE) {
        free_index(ix);
        tnn_set_error("non-finite or too large (|v| > 1e15) coordinate in input");
        return TNN_ERR_INVALID_ARG;
    }
    if (hm[META_FLAG] & BAD_ORDER) {
        free_index(ix);
        tnn_set_error("times are not sorted inside a trajectory");
        return TNN_ERR_INVALID_ARG;
    }
    memcpy(&ix->coord_max, &hm[1], sizeof(float));
    for (int d = 0; d < 4; ++d) {
        ix->bb_lo[d] = host_ord2f(hm[2 + 2 * d]);
        ix->bb_hi[d] = host_ord2f(hm[3 + 2 * d]);
    }
    double dur = 0.0;
    memcpy(&dur, &hm[10], sizeof(double));
    const GridBuild geo = grid_geometry(q0 * ix->bb_lo[0], q0 * ix->bb_hi[0], q1 * ix->bb_lo[1],
                                        q1 * ix->bb_hi[1], ix->bb_lo[3], ix->bb_hi[3], dur, S);

    // ---- the grid-key sort and, after the fit, the grid's per-key aggregates
    // on the second side stream; the t_A order and the running maximum of t_B
    // on `st`; all join before the grid's offsets and records
    e = cudaStreamWaitEvent(side[1], ev.e[0], 0);
    if (e == cudaSuccess) {
        k_grid_sort_keys<<<(s2 + tb - 1) / tb, tb, 0, side[1]>>>(ix->pts, range, Si, s2, q0, q1, geo, keys2);
        int bits = 1;
        while ((1ll << bits) - 1 < (long long)geo.nb * geo.ncell) // all ones stays free for the padding
            ++bits;
        if (sort_by_value(keys2, s2, bits, side[1]) != TNN_OK)
            e = cudaErrorUnknown;
    }
    tnn_status gs = e == cudaSuccess ? grid_alloc(ix, geo, st) : TNN_ERR_CUDA;
    if (gs == TNN_OK) {
        e = cudaEventRecord(ev.e[4], st); // the fit and the grid's zeroed arrays
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(side[1], ev.e[4], 0);
        if (e == cudaSuccess) {
            k_grid_extents<<<(Si + 127) / 128, 128, 0, side[1]>>>(
                rec, Si, geo, (unsigned int *)ix->g_ext, (unsigned int *)ix->g_tB, (unsigned int *)ix->g_bpm);
            e = cudaEventRecord(ev.e[3], side[1]);
        }
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(st, ev.e[2], 0);
        if (e == cudaSuccess) {
            k_gather_segments<<<nblk, 1024, 0, st>>>(keys, rec, Si, ix->seg, ix->segTA, pos, bmax);
            k_pm_apply<<<nblk, 1024, 0, st>>>(ix->seg, Si, bmax, ix->segPM);
            e = cudaStreamWaitEvent(st, ev.e[3], 0);
        }
        gs = e == cudaSuccess ? build_grid(ix, keys2, rec, pos, geo, st) : TNN_ERR_CUDA;
    }
    if (gs != TNN_OK) {
        if (e != cudaSuccess)
            tnn_set_error("index build failed: %s", cudaGetErrorString(e));
        free_index(ix); // waits for the device, the side streams included
        return gs;
    }
    // The build runs on after this call returns (stream order); a failure
    // there surfaces at the next synchronising call.
    e = cudaEventRecord(ix->built, st);
    if (e == cudaSuccess)
        e = cudaGetLastError();
    if (e != cudaSuccess) {
        free_index(ix);
        tnn_set_error("index build failed: %s", cudaGetErrorString(e));
        return TNN_ERR_CUDA;
    }
    *out = ix;
    return TNN_OK;
}

extern "C" void tnn_index_destroy(tnn_index *index) { free_index(index); }

static std::mutex g_time_order_mu;

tnn_status tnn_index_time_order(const tnn_index *cix, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(g_time_order_mu);
    tnn_index *ix = const_cast<tnn_index *>(cix);
    if (ix->pts_t)
        return TNN_OK;
    const int n = (int)ix->n, n2 = tnn_next_pow2_sort(n), tb = 256;
    float4 *pts_t = nullptr;
    int32_t *idx_t = nullptr;
    DevBuf keys_d;
    cudaError_t e = tnn_alloc((void **)&pts_t, sizeof(float4) * n, st);
    if (e == cudaSuccess)
        e = tnn_alloc((void **)&idx_t, sizeof(int32_t) * (n + 4), st); // padding for 16-byte copies
    if (e == cudaSuccess)
        e = keys_d.alloc(sizeof(unsigned long long) * n2, st);
    if (e != cudaSuccess) {
        tnn_free(pts_t, st);
        tnn_free(idx_t, st);
        tnn_set_error("time-order allocation failed: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? TNN_ERR_OOM : TNN_ERR_CUDA;
    }
    unsigned long long *keys = (unsigned long long *)keys_d.p;
    k_time_keys<<<(n2 + tb - 1) / tb, tb, 0, st>>>(ix->pts, n, keys, n2);
    tnn_bitonic_sort(keys, n2, st);
    k_gather_points<<<(n + tb - 1) / tb, tb, 0, st>>>(keys, ix->pts, n, pts_t, idx_t);
    e = cudaMemsetAsync(idx_t + n, 0, 4 * sizeof(int32_t), st);
    if (e == cudaSuccess)
        e = cudaGetLastError();
    if (e != cudaSuccess) {
        tnn_free(pts_t, st);
        tnn_free(idx_t, st);
        tnn_set_error("time order failed: %s", cudaGetErrorString(e));
        return TNN_ERR_CUDA;
    }
    ix->pts_t = pts_t;
    ix->idx_t = idx_t;
    return TNN_OK;
}

// ------------------------------------------------------------ space order

__global__ void k_space_keys(const float4 *__restrict__ p, int n, float4 lo, float4 sc,
                             unsigned long long *__restrict__ keys, int n2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        keys[i] = ((unsigned long long)tnn_morton_xyt(p[i], lo, sc) << 32) | (unsigned)i;
    else if (i < n2)
        keys[i] = ~0ull;
}

__global__ void k_gather_space(const unsigned long long *__restrict__ keys, const float4 *__restrict__ p,
                               int n, float4 *__restrict__ pm, int32_t *__restrict__ im,
                               uint32_t *__restrict__ cm)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const unsigned long long k = keys[i];
        const int j = (int)(k & 0xffffffffull);
        pm[i] = p[j];
        im[i] = j;
        cm[i] = (uint32_t)(k >> 32);
    }
}

static std::mutex g_space_order_mu;

tnn_status tnn_index_space_order(const tnn_index *cix, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(g_space_order_mu);
    tnn_index *ix = const_cast<tnn_index *>(cix);
    if (ix->pts_m)
        return TNN_OK;
    const int n = (int)ix->n, n2 = tnn_next_pow2_sort(n), tb = 256;
    float4 *pm = nullptr;
    int32_t *im = nullptr;
    uint32_t *cm = nullptr;
    DevBuf keys_d;
    cudaError_t e = tnn_alloc((void **)&pm, sizeof(float4) * n, st);
    if (e == cudaSuccess)
        e = tnn_alloc((void **)&im, sizeof(int32_t) * n, st);
    if (e == cudaSuccess)
        e = tnn_alloc((void **)&cm, sizeof(uint32_t) * n, st);
    if (e == cudaSuccess)
        e = keys_d.alloc(sizeof(unsigned long long) * n2, st);
    if (e != cudaSuccess) {
        tnn_free(pm, st);
        tnn_free(im, st);
        tnn_free(cm, st);
        tnn_set_error("space-order allocation failed: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? TNN_ERR_OOM : TNN_ERR_CUDA;
    }
    float4 l4, s4;
    tnn_morton_frame(ix->bb_lo, ix->bb_hi, &l4, &s4);
    unsigned long long *keys = (unsigned long long *)keys_d.p;
    k_space_keys<<<(n2 + tb - 1) / tb, tb, 0, st>>>(ix->pts, n, l4, s4, keys, n2);
    tnn_bitonic_sort(keys, n2, st);
    k_gather_space<<<(n + tb - 1) / tb, tb, 0, st>>>(keys, ix->pts, n, pm, im, cm);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        tnn_free(pm, st);
        tnn_free(im, st);
        tnn_free(cm, st);
        tnn_set_error("space order failed: %s", cudaGetErrorString(e));
        return TNN_ERR_CUDA;
    }
    ix->pts_m = pm;
    ix->idx_m = im;
    ix->code_m = cm;
    return TNN_OK;
}

// ------------------------------------------------------------- key order

// Padded run length of every key: its segments' member count rounded up to
// a multiple of 4 (so every run starts on a 16-byte boundary of idx_k).
__global__ void k_key_runs(const int32_t *__restrict__ off, const float4 *__restrict__ gseg, int nkeys,
                           int64_t *__restrict__ len)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nkeys)
        return;
    int64_t c = 0;
    for (int i = off[k]; i < off[k + 1]; ++i)
        c += __float_as_int(gseg[4 * (size_t)i + 3].y);
    len[k] = (c + 3) & ~3ll;
}

// Exclusive prefix sum of n int64 values by one block, in place, with the
// total appended at v[n] (n + 1 entries).
__global__ void __launch_bounds__(1024) k_scan_i64(int64_t *__restrict__ v, int n)
{
    __shared__ int64_t part[1024];
    const int per = (n + 1023) / 1024;
    const int lo = min(n, (int)threadIdx.x * per), hi = min(n, lo + per);
    int64_t s = 0;
    for (int i = lo; i < hi; ++i)
        s += v[i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int64_t a = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += a;
        __syncthreads();
    }
    int64_t run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int i = lo; i < hi; ++i) {
        const int64_t x = v[i];
        v[i] = run;
        run += x;
    }
    if (threadIdx.x == 1023)
        v[n] = part[1023];
}

// Every key's members into its run, then the padding.
__global__ void k_key_gather(const int32_t *__restrict__ off, const float4 *__restrict__ gseg,
                             const int64_t *__restrict__ start, int nkeys, const float4 *__restrict__ pts,
                             float4 *__restrict__ pk, int32_t *__restrict__ ik, int32_t *__restrict__ ks)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > nkeys)
        return;
    ks[k] = (int32_t)start[k];
    if (k == nkeys)
        return;
    int64_t o = start[k];
    float4 first = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = off[k]; i < off[k + 1]; ++i) {
        const float4 r = gseg[4 * (size_t)i + 3];
        const int f = __float_as_int(r.x), c = __float_as_int(r.y);
        if (i == off[k])
            first = pts[f];
        for (int j = 0; j < c; ++j, ++o) {
            pk[o] = pts[f + j];
            ik[o] = f + j;
        }
    }
    for (; o < start[k + 1]; ++o) {
        pk[o] = first;
        ik[o] = -1;
    }
}

static std::mutex g_key_order_mu;

tnn_status tnn_index_key_order(const tnn_index *cix, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(g_key_order_mu);
    tnn_index *ix = const_cast<tnn_index *>(cix);
    if (ix->pts_k)
        return TNN_OK;
    const int nkeys = ix->grid.nb * ix->grid.ncell, tb = 256;
    DevBuf len_d;
    TNN_CUDA_TRY(len_d.alloc(sizeof(int64_t) * (nkeys + 1), st));
    int64_t *len = (int64_t *)len_d.p;
    k_key_runs<<<(nkeys + tb - 1) / tb, tb, 0, st>>>(ix->g_off, ix->g_seg, nkeys, len);
    k_scan_i64<<<1, 1024, 0, st>>>(len, nkeys);
    int64_t nk = 0;
    TNN_CUDA_TRY(cudaMemcpyAsync(&nk, len + nkeys, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    TNN_CUDA_TRY(cudaStreamSynchronize(st));
    if (nk >= (1ll << 31) - 256) {
        tnn_set_error("the key-ordered copy (%lld points with padding) exceeds 2^31", (long long)nk);
        return TNN_ERR_UNSUPPORTED;
    }
    float4 *pk = nullptr;
    int32_t *ik = nullptr, *ks = nullptr;
    cudaError_t e = tnn_alloc((void **)&pk, sizeof(float4) * (size_t)std::max<int64_t>(nk, 1), st);
    if (e == cudaSuccess)
        e = tnn_alloc((void **)&ik, sizeof(int32_t) * (size_t)(nk + 4), st);
    if (e == cudaSuccess)
        e = tnn_alloc((void **)&ks, sizeof(int32_t) * (size_t)(nkeys + 1), st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(ik + nk, 0xff, 4 * sizeof(int32_t), st);
    if (e == cudaSuccess) {
        k_key_gather<<<(nkeys + 1 + tb - 1) / tb, tb, 0, st>>>(ix->g_off, ix->g_seg, len, nkeys, ix->pts, pk,
                                                             ik, ks);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        tnn_free(pk, st);
        tnn_free(ik, st);
        tnn_free(ks, st);
        tnn_set_error("key order failed: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? TNN_ERR_OOM : TNN_ERR_CUDA;
    }
    ix->pts_k = pk;
    ix->idx_k = ik;
    ix->kp_start = ks;
    ix->nk = nk;
    return TNN_OK;
}

extern "C" tnn_status tnn_index_get_info(const tnn_index *ix, tnn_index_info *out)
{
    tnn_clear_error();
    TNN_ARG_CHECK(ix && out, "NULL argument");
    out->n_points = ix->n;
    out->n_traj = ix->n_traj;
    out->n_segments = ix->S;
    out->seg_len = ix->K;
    out->coord_max = ix->coord_max;
    if (!ix->rmax_known) {
        // the segment fit's largest radius: wait for the build to finish
        static std::mutex mu;
        std::lock_guard<std::mutex> lk(mu);
        tnn_index *w = const_cast<tnn_index *>(ix);
        unsigned int bits = 0u;
        cudaError_t e = ix->built ? cudaEventSynchronize(ix->built) : cudaSuccess;
        if (e == cudaSuccess)
            e = cudaMemcpy(&bits, ix->d_rmax, sizeof(bits), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) {
            tnn_set_error("reading the index radius failed: %s", cudaGetErrorString(e));
            return TNN_ERR_CUDA;
        }
        memcpy(&w->max_radius, &bits, sizeof(float));
        w->rmax_known = true;
    }
    out->max_radius = ix->max_radius;
    return TNN_OK;
}

extern "C" tnn_status tnn_index_export(const tnn_index *ix, float *d_seg,
                                       float *d_pm, tnn_stream_t stream)
{
    tnn_clear_error();
    TNN_ARG_CHECK(ix && d_seg, "NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    TNN_CUDA_TRY(cudaMemcpyAsync(d_seg, ix->seg, sizeof(float4) * 4 * ix->S,
                                 cudaMemcpyDeviceToDevice, st));
    if (d_pm)
        TNN_CUDA_TRY(cudaMemcpyAsync(d_pm, ix->segPM, sizeof(float) * ix->S,
                                     cudaMemcpyDeviceToDevice, st));
    return TNN_OK;
}
