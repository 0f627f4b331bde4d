// Nearest centre of many points: argmin over centres of the fp64 squared distance (dimensions in increasing
// order, multiply and add rounded separately; ties to the smaller centre index), without evaluating most of
// the fp64 distances.
//
// A centre is rounded to a 16-bit vector `hi` (the points' element type); m = |c - hi|. With x.hi from tensor cores,
//   s_c = |c|^2 - 2 x.hi      (the squared distance less |x|^2, the same for every centre)
// orders the centres up to an error: what the rounding leaves out is at most 2 |x| m, eight MMAs of 16 values in a
// row cost at most 8 * 17 * 2^-23 of sum |x_d hi_d| <= (1 + 2^-8) (|x|^2 + |c|^2) / 2 (see select_rows.cuh): together at most
// E_c = kNearErr (|x|^2 + |c|^2) + 2 |x| m. The scan keeps, per point, the smallest upper bound so far, and of the centres
// whose lower bound does not exceed it the three smallest lower bounds with their centres and the fourth smallest.
// Usually one is left at the end; where two or three are, they are compared in fp64, where there are more all centres
// are (with early exit). (A second product with c - hi would leave fewer open, for twice the MMAs. Keeping the
// smallest lower bounds whatever the upper one took 79 us instead of 70 for 4 x 4096 points and 2048 centres:
// every centre was inserted somewhere in a warp.) Products that underflow fp32 add less than 1e-34.
#pragma once
#include <math_constants.h>

#include "common.cuh"
#include "select_rows.cuh"

namespace santapp {

constexpr float kNearErr = 2.2e-5f;
constexpr int kNearPoints = 256;         // points per block
constexpr int kNearThreads = 256;        // 8 warps of 32 points
constexpr int kNearTile = 64;            // centres per shared-memory stage

// Bounds leave out what all centres of a point share (its kNearErr |x|^2): lower s_c - kNearErr |c|^2 - 2 |x| m, and the
// upper bound with that part counted twice.
struct NearTop {                         // smallest lower bounds of a point, their centres, the fourth smallest; the smallest upper bound
    float t1, t2, t3, t4, upper;
    int i1, i2, i3;
};
static_assert(sizeof(NearTop) == kNearTopBytes, "the fit's workspace holds these");
__device__ __forceinline__ NearTop near_none(int i)
{
    return {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, i, i, i};
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
__device__ __forceinline__ bool near_open(const NearTop &n, float nx) { return !(nx <= 1e37f) || !(fabsf(n.t1) < CUDART_INF_F) || !(n.t4 > n.upper); }

// A centre with components beyond the element type, or whose squared norm fp32 cannot hold, is stored as zeros with
// a bound of -inf: it is a candidate of every point. Else: the lower bound's constant.
template <bool kHalf>
__device__ __forceinline__ float centre_bias(float nc) { return nc <= (kHalf ? 4.2e9f : 1e37f) ? nc * (1.f - kNearErr) : -CUDART_INF_F; }
template <bool kHalf>
__device__ __forceinline__ uint32_t pack_elems(float lo, float hi)
{
    uint32_t r;
    if constexpr (kHalf) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    else                 asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

struct NearSmem {
    uint4 ring[4][kNearTile * 16];       // stages (and, all of it, the points before the scan): rows of 256 bytes, 16-byte pieces XOR-swizzled
    float2 bias[2][kNearTile];           // constant of the lower bound, m
    float list[7][kNearThreads * 4];     // a thread's four points (of which it sees a quarter of the centres): t1 .. t4, i1 .. i3
    NearTop top[kNearPoints];
    float nx[kNearPoints];
};
__device__ __forceinline__ int near_piece(int row, int chunk) { return row * 16 + (chunk ^ (row & 7)); }

// The block's points as MMA operands: `row_of(i)` points to the 256 bytes of point i < kNearPoints (any valid
// row for a point past the end). Every thread of the block calls it.
template <bool kHalf, typename RowOf>
__device__ __forceinline__ void near_load_points(NearSmem &sm, RowOf row_of, uint32_t (&a)[2][8][4])
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint4 *rows = &sm.ring[0][0];                           // 64 KB: the whole ring
#pragma unroll 4
    for (int m = 0; m < 16; ++m) {                          // a warp copies its own 32 rows, two per step
        const int i = warp * 32 + 2 * m + (lane >> 4), ch = lane & 15;
        copy16_async(shared_addr(rows + near_piece(i, ch)), reinterpret_cast<const uint4 *>(row_of(i)) + ch);
    }
    copy_async_wait();
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int s = 0; s < 8; ++s)
            ldmatrix4(a[m][s], shared_addr(rows + near_piece(warp * 32 + 16 * m + (lane & 15), 2 * s + (lane >> 4))));
    // squared norms, from the fragments: rows g and g + 8 of each group of 16
    float n[2][2];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        n[m][0] = n[m][1] = 0.f;
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float x0 = elem_lo<kHalf>(a[m][s][r]), x1 = elem_hi<kHalf>(a[m][s][r]);
                n[m][r & 1] = fmaf(x0, x0, fmaf(x1, x1, n[m][r & 1]));
            }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            n[m][h] += __shfl_xor_sync(0xFFFFFFFFu, n[m][h], 1);
            n[m][h] += __shfl_xor_sync(0xFFFFFFFFu, n[m][h], 2);
            if ((lane & 3) == 0) sm.nx[warp * 32 + 16 * m + 8 * h + (lane >> 2)] = n[m][h];
        }
    __syncthreads();                                        // the ring is free
}

// The scan over centres [k_lo, k_hi): `fill(stage, base, n)` brings centres [base, base + n) into a stage
// (asynchronous copies of it are waited for here). Leaves the points' NearTop in sm.top.
template <bool kHalf, typename Fill>
__device__ __forceinline__ void near_scan(NearSmem &sm, const uint32_t (&a)[2][8][4], int k_lo, int k_hi, Fill fill)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane & 3;
    // The thread's points are rows g, g + 8, g + 16, g + 24 of the warp's 32. Their lists are in shared memory: they are
    // touched rarely, and would not fit in registers beside the points.
    float reach[4], shared[4], upper[4];                    // 2 |x|, the part of the upper bound that all centres share
    auto slot = [&](int r) { return &sm.list[0][r * kNearThreads + threadIdx.x]; };
    constexpr int kWord = kNearThreads * 4;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float *l = slot(r);
#pragma unroll
        for (int w = 0; w < 4; ++w) l[w * kWord] = CUDART_INF_F;
#pragma unroll
        for (int w = 4; w < 7; ++w) l[w * kWord] = __int_as_float(k_lo);
        const float nx = sm.nx[warp * 32 + 8 * r + (lane >> 2)];
        reach[r] = 2.000002f * sqrtf(nx);
        shared[r] = fmaf(2.f * kNearErr, nx, 1e-34f);
        upper[r] = CUDART_INF_F;
    }
    auto load = [&](int r) {
        const float *l = slot(r);
        return NearTop{l[0], l[kWord], l[2 * kWord], l[3 * kWord], upper[r], __float_as_int(l[4 * kWord]), __float_as_int(l[5 * kWord]),
                       __float_as_int(l[6 * kWord])};
    };
    auto insert = [&](int r, float s, int i) {
        NearTop n = load(r);
        near_insert(n, s, i);
        float *l = slot(r);
        l[0] = n.t1;
        l[kWord] = n.t2;
        l[2 * kWord] = n.t3;
        l[3 * kWord] = n.t4;
        l[4 * kWord] = __int_as_float(n.i1);
        l[5 * kWord] = __int_as_float(n.i2);
        l[6 * kWord] = __int_as_float(n.i3);
    };
    fill(0, k_lo, min(kNearTile, k_hi - k_lo));
    asm volatile("cp.async.commit_group;");
    int stage = 0;
    for (int base = k_lo; base < k_hi; base += kNearTile, stage ^= 1) {
        if (base + kNearTile < k_hi) fill(stage ^ 1, base + kNearTile, min(kNearTile, k_hi - base - kNearTile));
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const uint32_t hi_a = shared_addr(&sm.ring[stage][0]);
#pragma unroll 2
        for (int nt = 0; nt < kNearTile / 8; ++nt) {
            float acc[2][2][4];                             // two chains of four MMAs each per group of 16 points
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) acc[m][h][0] = acc[m][h][1] = acc[m][h][2] = acc[m][h][3] = 0.f;
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) {
                uint32_t bh[4];
                ldmatrix4(bh, hi_a + (uint32_t)near_piece(nt * 8 + (lane & 7), 4 * s2 + (lane >> 3)) * 16u);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint32_t(&f)[4] = a[m][2 * s2 + h];
                        mma_rows<kHalf>(acc[m][h], f[0], f[1], f[2], f[3], bh[2 * h], bh[2 * h + 1]);
                    }
            }
            const float4 bias = *reinterpret_cast<const float4 *>(&sm.bias[stage][nt * 8 + 2 * c]);
            float low[2][4];
            bool some = false;
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = 2 * m + (e >> 1);
                    low[m][e] = fmaf(-2.f, acc[m][0][e] + acc[m][1][e], fmaf(-reach[r], (e & 1) ? bias.w : bias.y, (e & 1) ? bias.z : bias.x));
                    some |= low[m][e] < upper[r];
                }
            if (some) {
                const int col = base + nt * 8 + 2 * c;
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int r = 2 * m + (e >> 1);
                        if (low[m][e] < upper[r]) {
                            // (1.0001: the stored constant is |c|^2 (1 - kNearErr), rounded)
                            const float wide = fmaf(1.0001f * kNearErr, (e & 1) ? bias.z : bias.x, reach[r] * ((e & 1) ? bias.w : bias.y));
                            upper[r] = fminf(upper[r], fmaf(2.f, wide, low[m][e] + shared[r]));
                            insert(r, low[m][e], col + (e & 1));
                        }
                    }
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {                       // the four lanes of a point share its upper bound
            upper[r] = fminf(upper[r], __shfl_xor_sync(0xFFFFFFFFu, upper[r], 1));
            upper[r] = fminf(upper[r], __shfl_xor_sync(0xFFFFFFFFu, upper[r], 2));
        }
        __syncthreads();                                    // the stage may be filled again
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        NearTop top = load(r);
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            NearTop n;
            n.t1 = __shfl_xor_sync(0xFFFFFFFFu, top.t1, o);
            n.t2 = __shfl_xor_sync(0xFFFFFFFFu, top.t2, o);
            n.t3 = __shfl_xor_sync(0xFFFFFFFFu, top.t3, o);
            n.t4 = __shfl_xor_sync(0xFFFFFFFFu, top.t4, o);
            n.upper = top.upper;
            n.i1 = __shfl_xor_sync(0xFFFFFFFFu, top.i1, o);
            n.i2 = __shfl_xor_sync(0xFFFFFFFFu, top.i2, o);
            n.i3 = __shfl_xor_sync(0xFFFFFFFFu, top.i3, o);
            near_merge(top, n);
        }
        if (c == 0) sm.top[warp * 32 + 8 * r + (lane >> 2)] = top;
    }
    __syncwarp();                                           // a warp's points are its own rows
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
