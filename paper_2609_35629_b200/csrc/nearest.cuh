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
// smallest upper bound; where that leaves two or three they are compared in fp64, where it leaves more all
// centres are (with early exit). Products that underflow fp32 add less than kUnderflow.
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
    for (int i = 0; i < (1 << 20); ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(done) : "r"(shared_addr(&sm.done[buf])), "r"(parity) : "memory");
        if (done) return;
    }
    sm.failed = 1;
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

// All centres in fp64, one point per warp (a lane takes every 32nd centre): for points the bounds leave open.
// A lane gives a centre up once its partial sum exceeds the best so far (sums only grow). Every lane gets the
// result; like the plain loop, distances that are not smaller than infinity leave centre 0.
template <bool kHalf, typename C>
__device__ __noinline__ int near_scan_exact(const uint4 *x, const C *cen, int k, double &dist)
{
    const int lane = threadIdx.x & 31;
    double best = CUDART_INF;
    int arg = INT_MAX;
    for (int u = lane; u < k; u += 32) {
        const C *cu = cen + (size_t)u * kHeadDim;
        double s = 0.0;
        for (int q = 0; q < 16 && !(s > best); ++q) {
            const uint4 w4 = __ldg(x + q);
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const double e0 = __dsub_rn((double)elem_lo<kHalf>(w[t]), (double)cu[8 * q + 2 * t]);
                const double e1 = __dsub_rn((double)elem_hi<kHalf>(w[t]), (double)cu[8 * q + 2 * t + 1]);
                s = __dadd_rn(s, __dmul_rn(e0, e0));
                s = __dadd_rn(s, __dmul_rn(e1, e1));
            }
        }
        if (s < best) { best = s; arg = u; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const int j = __shfl_xor_sync(0xFFFFFFFFu, arg, o);
        if (w < best || (w == best && j < arg)) { best = w; arg = j; }
    }
    dist = best;
    return arg == INT_MAX ? 0 : arg;
}

}  // namespace santapp
