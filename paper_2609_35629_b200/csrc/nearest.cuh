// Nearest centre of many points: argmin over centres of the fp64 squared distance (dimensions in increasing
// order, multiply and add rounded separately; ties to the smaller centre index), without evaluating most of
// the fp64 distances.
//
// A centre is rounded to a 16-bit vector `hi` (the points' element type); m = |c - hi|. With x.hi from tensor cores,
//   s_c = |c|^2 - 2 x.hi      (the squared distance less |x|^2, the same for every centre)
// orders the centres up to an error: what the rounding leaves out is at most 2 |x| m; eight MMAs of 16 values in a
// row cost at most 8 * 17 * 2^-23 of sum |x_d hi_d| <= (1 + 2^-8) (|x|^2 + |c|^2) / 2 (see select_rows.cuh), twice that for the
// distance; the column of a centre, kept in the last five bits of its bound, 2^-18 of at most 2.04 (|x|^2 + |c|^2).
// Together at most E_c = kNearErr (|x|^2 + |c|^2) + 2 |x| m. A centre can be nearest only if its lower bound does not exceed the
// smallest upper bound; where that leaves two or three they are compared in fp64, where it leaves more the
// point goes through all centres (near_scan_exact, near_scan_tiles). Products that underflow fp32 add less than kUnderflow.
//
// The products are a GEMM (tcgen05, 128 points x 128 centres x 128 dimensions a tile, 512 cycles at the measured rate);
// looking at 16384 results takes the block's eight warps about twice that, since every one costs two FMAs and four
// minimum or logic operations at half rate, so two blocks share an SM and the tensor core is busy half the time. The
// search is free of branches over a chunk of 32 centres (its two smallest bounds), because in a warp of 32
// points some lane would take any branch that a new minimum takes: mma.sync with such a branch per value took
// 70 us for 4 x 4096 points and 2048 centres, this 37.
#pragma once
#include <math_constants.h>

#include "common.cuh"
#include "select_rows.cuh"
#include "tc.cuh"

namespace santapp {

constexpr float kNearErr = 3.0e-5f;
constexpr float kNearFar = 3.0e38f;      // a bound that says nothing: below -1e38, all centres have to be compared; above 1e38, no centre
constexpr int kNearPoints = 128;         // points per block: the rows of an accumulator
constexpr int kNearThreads = 256;        // warps w and w + 4 look at the two halves of the columns of points 32 (w & 3) ..
constexpr int kNearTile = 128;           // centres per shared-memory stage: the columns

// Bounds leave out what all centres of a point share (its kNearErr |x|^2): lower s_c - kNearErr |c|^2 - 2 |x| m, and the
// upper bound with that part counted twice.
struct NearTop {                         // smallest lower bounds of a point, their centres, the fourth smallest; the smallest upper bound
    float t1, t2, t3, t4, upper;
    int i1, i2, i3;
};
static_assert(sizeof(NearTop) == kNearTopBytes, "the fit's workspace holds these");
__device__ __forceinline__ NearTop near_none(int i)
{
    return {kNearFar, kNearFar, kNearFar, kNearFar, kNearFar, i, i, i};
}
__device__ __forceinline__ void near_insert(NearTop &n, float s, int i)
{
    if (s < n.t4) {
        if (s < n.t3) {
            n.t4 = n.t3;
            if (s < n.t2) {
                n.t3 = n.t2; n.i3 = n.i2;
                if (s < n.t1) { n.t2 = n.t1; n.i2 = n.i1; n.t1 = s; n.i1 = i; }
                else { n.t2 = s; n.i2 = i; }
            } else {
                n.t3 = s; n.i3 = i;
            }
        } else {
            n.t4 = s;
        }
    }
}
__device__ __forceinline__ void near_merge(NearTop &n, const NearTop &o)
{
    near_insert(n, o.t1, o.i1);
    near_insert(n, o.t2, o.i2);
    near_insert(n, o.t3, o.i3);
    if (o.t4 < n.t4) n.t4 = o.t4;        // not below n.t3: the three before it have been inserted
    n.upper = fminf(n.upper, o.upper);
}
// Whether the bounds say too little, and all centres have to be compared.
__device__ __forceinline__ bool near_open(const NearTop &n, float nx) { return !(nx <= 1e37f) || !(fabsf(n.t1) < 1e38f) || !(n.t4 > n.upper); }

// A centre with components beyond the element type, or whose squared norm fp32 cannot hold, is stored as zeros with
// a bound of -kNearFar: every point compares all centres. Else: the lower bound's constant.
template <bool kHalf>
__device__ __forceinline__ float centre_bias(float nc) { return nc <= (kHalf ? 4.2e9f : 1e37f) ? nc * (1.f - kNearErr) : -kNearFar; }
template <bool kHalf>
__device__ __forceinline__ uint32_t pack_elems(float lo, float hi)
{
    uint32_t r;
    if constexpr (kHalf) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    else                 asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

struct NearSmem {
    // K-major operands with the tensor core's 128-byte swizzle (near_byte)
    alignas(1024) unsigned char points[kNearPoints * 256];
    unsigned char centres[2][kNearTile * 256];
    float2 bias[3][kNearTile];           // constant of the lower bound and m, by tile
    float nx[kNearPoints];
    int idx[kNearPoints];                // for the caller: tokens of the points
    NearTop top[kNearPoints];
    uint64_t done[2];                    // mbarriers: the products in an accumulator buffer are there
    uint32_t tmem;
    int failed;                          // a wait ran out (never expected): all centres are compared
};
static_assert(kNearTile == kNearPoints, "both operands have one layout");
// Byte of 16-byte piece ch of row r: atoms of 64 values of eight rows, pieces XOR-swizzled inside.
__device__ __forceinline__ int near_byte(int r, int ch) { return (ch >> 3) * (kNearPoints * 128) + (r >> 3) * 1024 + (r & 7) * 128 + (((ch & 7) ^ (r & 7)) << 4); }
__device__ __forceinline__ void copy16_or_zero(uint32_t dst, const void *src, bool real)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(real ? 16 : 0) : "memory");
}

// Tensor memory (two accumulator buffers of kNearTile columns) and barriers; every thread of the block, at its
// beginning and its end.
__device__ __forceinline__ void near_open_block(NearSmem &sm)
{
    if (threadIdx.x == 0) {
        sm.failed = 0;
        for (int i = 0; i < 2; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(shared_addr(&sm.done[i])), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(shared_addr(&sm.tmem)), "r"(2 * kNearTile) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}
__device__ __forceinline__ void near_close_block(NearSmem &sm)
{
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(2 * kNearTile));
}
__device__ __forceinline__ void near_wait(NearSmem &sm, int buf, uint32_t parity)
{
    if (*reinterpret_cast<volatile int *>(&sm.failed)) return;
    if (!tc_wait(shared_addr(&sm.done[buf]), parity)) sm.failed = 1;
}

// One point against 32 consecutive centres from `first` on: v their products with it, bias their constants.
__device__ __forceinline__ void near_look(NearTop &n, const uint32_t (&v)[32], const float2 *bias, int first, float reach, float shared)
{
    float key[32], t1 = kNearFar, t2 = kNearFar;
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        const float4 b = *reinterpret_cast<const float4 *>(bias + c);
        const float l0 = fmaf(-2.f, __uint_as_float(v[c]), fmaf(-reach, b.y, b.x));
        const float l1 = fmaf(-2.f, __uint_as_float(v[c + 1]), fmaf(-reach, b.w, b.z));
        key[c] = __uint_as_float((__float_as_uint(l0) & ~31u) | (uint32_t)c);
        key[c + 1] = __uint_as_float((__float_as_uint(l1) & ~31u) | (uint32_t)(c + 1));
        t2 = fminf(t2, fmaxf(t1, key[c]));
        t1 = fminf(t1, key[c]);
        t2 = fminf(t2, fmaxf(t1, key[c + 1]));
        t1 = fminf(t1, key[c + 1]);
    }
    if (t1 <= n.upper) {
        const float2 b = bias[__float_as_uint(t1) & 31u];
        // (1.0001: the stored constant is |c|^2 (1 - kNearErr), rounded. The mark of a centre that the products say nothing about
        // bounds nothing from above: it stays the smallest key, and near_open finds it.)
        if (t1 > -1e38f) n.upper = fminf(n.upper, fmaf(2.f, fmaf(1.0001f * kNearErr, b.x, reach * b.y), t1 + shared));
        near_insert(n, t1, first + (int)(__float_as_uint(t1) & 31u));
    }
    while (__any_sync(0xFFFFFFFFu, t2 <= n.upper)) {         // some point of the warp has another candidate here
        if (t2 <= n.upper) near_insert(n, t2, first + (int)(__float_as_uint(t2) & 31u));
        float next = kNearFar;
#pragma unroll
        for (int c = 0; c < 32; ++c) next = fminf(next, key[c] > t2 ? key[c] : kNearFar);
        t2 = next < kNearFar ? next : CUDART_INF_F;
    }
}

// The nearest centres among [k_lo, k_hi) of the block's points, left in sm.top (for all threads to read). `row_of(i)`
// points to the 256 bytes of point i < kNearPoints (any valid row for a point past the end); `fill(stage, slot, base, n)`
// brings centres [base, base + n) into a stage and their constants into a slot of the bias table, by asynchronous copies
// or plain stores, with zeros and kNearFar behind them. `uses`: how often the accumulator buffers have been
// waited for, kept by the caller, 0 at first.
template <bool kHalf, typename RowOf, typename Fill>
__device__ __forceinline__ void near_scan(NearSmem &sm, RowOf row_of, int k_lo, int k_hi, uint32_t (&uses)[2], Fill fill)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_tiles = (k_hi - k_lo + kNearTile - 1) / kNearTile, row = 32 * (warp & 3) + lane;
    fill(0, 0, k_lo, min(kNearTile, k_hi - k_lo));
#pragma unroll
    for (int m = 0; m < kNearPoints * 16 / kNearThreads; ++m) {
        const int e = m * kNearThreads + tid;
        copy16_async(shared_addr(sm.points + near_byte(e >> 4, e & 15)), reinterpret_cast<const uint4 *>(row_of(e >> 4)) + (e & 15));
    }
    NearTop top = near_none(k_lo);
    float reach = 0.f, shared = 0.f;                        // 2 |x|, the part of the upper bound that all centres share
    for (int i = 0; i <= n_tiles; ++i) {
        if (i < n_tiles) {
            copy_async_wait();
            proxy_fence();
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (i < n_tiles && tid == 0) {
            const uint64_t da = tc_desc_sw128(shared_addr(sm.points), 16, 1024), db = tc_desc_sw128(shared_addr(sm.centres[i & 1]), 16, 1024);
            const uint32_t idesc = tc_idesc(kNearPoints, kNearTile, 0, 0, kHalf);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const uint64_t at = (uint64_t)(((s >> 2) * (kNearPoints * 128) + (s & 3) * 32) >> 4);
                tc_mma(sm.tmem + kNearTile * (i & 1), da + at, db + at, idesc, s > 0 ? 1u : 0u);
            }
            tc_commit(shared_addr(&sm.done[i & 1]));
        }
        if (i == 0) {                                       // beside the first product: the points' norms
            float n = 0.f;
#pragma unroll 4
            for (int ch = 0; ch < 16; ++ch) {
                const uint4 w4 = *reinterpret_cast<const uint4 *>(sm.points + near_byte(row, ch));
                const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float x0 = elem_lo<kHalf>(w[t]), x1 = elem_hi<kHalf>(w[t]);
                    n = fmaf(x0, x0, fmaf(x1, x1, n));
                }
            }
            if (warp < 4) sm.nx[row] = n;
            reach = 2.000002f * sqrtf(n);
            shared = fmaf(2.f * kNearErr, n, kUnderflow);
        } else {
            const int buf = (i - 1) & 1;
            near_wait(sm, buf, uses[buf] & 1u);
            ++uses[buf];
            tc_fence_after();
        }
        if (i + 1 < n_tiles) {                              // the product before this one has left the stage
            const int base = k_lo + (i + 1) * kNearTile;
            fill((i + 1) & 1, (i + 1) % 3, base, min(kNearTile, k_hi - base));
        }
        if (i > 0) {
            const int col = 64 * (warp >> 2);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
                tc_ld32(sm.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(kNearTile * ((i - 1) & 1) + col + 32 * half), v);
                near_look(top, v, sm.bias[(i - 1) % 3] + col + 32 * half, k_lo + (i - 1) * kNearTile + col + 32 * half, reach, shared);
            }
        }
    }
    if (sm.failed) top.t1 = -kNearFar;
    if (warp >= 4) sm.top[row] = top;
    __syncthreads();
    if (warp < 4) {
        near_merge(top, sm.top[row]);
        sm.top[row] = top;
    }
    __syncthreads();
}

// The defining distance of a point (128 packed 16-bit values) and a centre of doubles or floats.
template <bool kHalf, typename C>
__device__ __forceinline__ double near_exact(const uint4 *x, const C *cen)
{
    double s = 0.0;
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
        const uint4 w4 = __ldg(x + q);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double e0 = __dsub_rn((double)elem_lo<kHalf>(w[t]), (double)cen[8 * q + 2 * t]);
            const double e1 = __dsub_rn((double)elem_hi<kHalf>(w[t]), (double)cen[8 * q + 2 * t + 1]);
            s = __dadd_rn(s, __dmul_rn(e0, e0));
            s = __dadd_rn(s, __dmul_rn(e1, e1));
        }
    }
    return s;
}

// Four consecutive values of a centre (rows of floats need not be 16-byte aligned).
__device__ __forceinline__ void near_quad(const float *p, float (&v)[4])
{
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = __ldg(p + e);
    }
}
__device__ __forceinline__ void near_quad(const double *p, double (&v)[4])
{
    const double2 w0 = __ldg(reinterpret_cast<const double2 *>(p)), w1 = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = w0.x; v[1] = w0.y; v[2] = w1.x; v[3] = w1.y;
}

// All centres of one point by a warp, where the bounds leave few points of a block open. The centres come eight at a time,
// four dimensions per lane (whole lines; with a centre per lane a load touched 32). fp32 distances leave out
// most of them: a sum of (x - c)^2 whose c is rounded to fp32 once is off by at most 13 * 2^-24 of itself and 2^-23
// |x|^2. Of the rest, one equal to the best so far is no better, and the others are evaluated in fp64, terms by all
// lanes and then the sum in order. `term`: 128 doubles of the warp, 16-byte aligned. Every lane gets the result; like
// the plain loop, distances that are not smaller than infinity leave centre 0.
template <bool kHalf, typename C>
__device__ __noinline__ int near_scan_exact(const uint4 *x, const C *cen, int k, double *term, double &dist)
{
    const int lane = threadIdx.x & 31;
    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(x) + lane);
    const float xf[4] = {elem_lo<kHalf>(w.x), elem_hi<kHalf>(w.x), elem_lo<kHalf>(w.y), elem_hi<kHalf>(w.y)};
    const float slack = fmaf(1e-6f, warp_sum(fmaf(xf[0], xf[0], xf[1] * xf[1]) + fmaf(xf[2], xf[2], xf[3] * xf[3])), kUnderflow);
    const C *mine = cen + 4 * lane;
    double best = CUDART_INF;
    int arg = INT_MAX;
    C held[4] = {};                                         // the best centre's values
    float up = CUDART_INF_F;                                // no nearest centre is farther
    for (int base = 0; base < k; base += 8) {
        float d[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            C v[4];
            near_quad(mine + (size_t)min(base + c, k - 1) * kHeadDim, v);
            d[c] = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) d[c] = fmaf(xf[e] - (float)v[e], xf[e] - (float)v[e], d[c]);
        }
        // sums over the lanes, halving the centres a lane holds: lane l ends up with centre l >> 2
#pragma unroll
        for (int half = 4; half > 0; half >>= 1) {
            const bool upper = lane & (4 * half);
#pragma unroll
            for (int m = 0; m < half; ++m) d[m] = (upper ? d[m + half] : d[m]) + __shfl_xor_sync(0xFFFFFFFFu, upper ? d[m] : d[m + half], 4 * half);
        }
        d[0] += __shfl_xor_sync(0xFFFFFFFFu, d[0], 2);
        d[0] += __shfl_xor_sync(0xFFFFFFFFu, d[0], 1);
        const bool there = base + (lane >> 2) < k;
        up = fminf(up, __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(there ? fmaf(d[0], 2e-6f, d[0]) + slack : CUDART_INF_F))));
        for (unsigned left = __ballot_sync(0xFFFFFFFFu, there && (lane & 3) == 0 && !(fmaf(d[0], -2e-6f, d[0]) - slack > up)); left; left &= left - 1) {
            const int u = base + ((__ffs(left) - 1) >> 2);
            C v[4];
            near_quad(mine + (size_t)u * kHeadDim, v);
            if (arg != INT_MAX && __all_sync(0xFFFFFFFFu, v[0] == held[0] && v[1] == held[1] && v[2] == held[2] && v[3] == held[3])) continue;
            double t[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                t[e] = __dsub_rn((double)xf[e], (double)v[e]);
                t[e] = __dmul_rn(t[e], t[e]);
            }
            __syncwarp();
            *reinterpret_cast<double2 *>(term + 4 * lane) = make_double2(t[0], t[1]);
            *reinterpret_cast<double2 *>(term + 4 * lane + 2) = make_double2(t[2], t[3]);
            __syncwarp();
            double s = 0.0;
#pragma unroll 8
            for (int q = 0; q < kHeadDim; q += 2) {
                const double2 two = *reinterpret_cast<const double2 *>(term + q);
                s = __dadd_rn(s, two.x);
                s = __dadd_rn(s, two.y);
            }
            if (s < best) {
                best = s;
                arg = u;
#pragma unroll
                for (int e = 0; e < 4; ++e) held[e] = v[e];
            }
        }
    }
    __syncwarp();
    dist = best;
    return arg == INT_MAX ? 0 : arg;
}

// The same by a block for many open points (centres that repeat leave every point open), kShare threads per point: all
// fp64 distances, sixteen centres at a time as doubles in shared memory (`tile`, 16-byte aligned), eight of
// them per pass of a thread; a warp without open points only brings centres. Every thread of the block; `x` is
// a valid row in any case. The first kThreads / kShare threads get the results.
constexpr int kScanTile = 16;
template <bool kHalf, int kThreads, int kShare, typename C>
__device__ __noinline__ int near_scan_tiles(const uint4 *x, bool open, const C *cen, int k, double (*tile)[kHeadDim], double &dist)
{
    constexpr int kPoints = kThreads / kShare;
    const int tid = threadIdx.x, part = tid / kPoints;
    const bool busy = __any_sync(0xFFFFFFFFu, open);
    double best = CUDART_INF;
    int arg = INT_MAX;
    for (int base = 0; base < k; base += kScanTile) {
        __syncthreads();
        for (int e = tid; e < kScanTile * kHeadDim; e += kThreads)
            tile[e / kHeadDim][e % kHeadDim] = (double)__ldg(cen + (size_t)min(base + e / kHeadDim, k - 1) * kHeadDim + e % kHeadDim);
        __syncthreads();
        if (!busy) continue;
        for (int t = 8 * part; t < kScanTile; t += 8 * kShare) {
            const uint4 *const row[1] = {x};
            double d[1][8] = {};
            dist_points<kHalf, 1, 8, 8>(row, tile + t, d);
#pragma unroll
            for (int v = 0; v < 8; ++v)
                if (base + t + v < k && d[0][v] < best) { best = d[0][v]; arg = base + t + v; }
        }
    }
    __syncthreads();
    if constexpr (kShare == 2) {
        double *half_best = tile[0];
        int *half_arg = reinterpret_cast<int *>(tile[1]);
        if (part == 1) { half_best[tid - kPoints] = best; half_arg[tid - kPoints] = arg; }
        __syncthreads();
        if (part == 0 && (half_best[tid] < best || (half_best[tid] == best && half_arg[tid] < arg))) { best = half_best[tid]; arg = half_arg[tid]; }
    }
    dist = best;
    return arg == INT_MAX ? 0 : arg;
}

}  // namespace santapp
