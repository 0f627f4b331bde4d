// Nearest centre of many points: argmin over centres of the fp64 squared distance (dimensions in increasing
// order, multiply and add rounded separately; ties to the smaller centre index), without evaluating most of
// the fp64 distances.
//
// A centre is the sum of two 16-bit vectors, hi + mid (each component rounded twice to the points' element
// type: within 2^-17 of it), so x.c comes from tensor cores as two products, and
//   s_c = |c|^2 - 2 x.c      (the squared distance less |x|^2, the same for every centre)
// orders the centres up to an error. With S = sum |x_d c_d| <= (|x|^2 + |c|^2) / 2: eight MMAs of 16 values in a
// row cost at most 8 * 17 * 2^-23 S (see select_rows.cuh), what the split leaves out 2^-17 S, twice both: below
// kNearErr (|x|^2 + |c|^2). The scan keeps, per point, the two smallest lower bounds s_c - kNearErr |c|^2 with
// their centres and the third smallest; a centre whose lower bound exceeds the smallest by more than twice the
// error of that one cannot be nearest. Usually that leaves one; where it leaves two they are compared in
// fp64, where it leaves more all centres are (with early exit). fp16 halves below 2^-14 lose precision
// absolutely, which adds a term in |x|; products that underflow fp32 add less than 1e-34.
#pragma once
#include <math_constants.h>

#include "common.cuh"
#include "select_rows.cuh"

namespace santapp {

constexpr float kNearErr = 2.6e-5f;
constexpr int kNearPoints = 256;         // points per block
constexpr int kNearThreads = 256;        // 8 warps of 32 points
constexpr int kNearTile = 64;            // centres per shared-memory stage

struct NearTop {                         // smallest lower bounds of a point, their centres, the third smallest
    float t1, t2, t3;
    int i1, i2;
};
static_assert(sizeof(NearTop) == kNearTopBytes, "the fit's workspace holds these");
__device__ __forceinline__ void near_insert(NearTop &n, float s, int i)
{
    if (s < n.t3) {
        if (s < n.t2) {
            n.t3 = n.t2;
            if (s < n.t1) { n.t2 = n.t1; n.i2 = n.i1; n.t1 = s; n.i1 = i; }
            else { n.t2 = s; n.i2 = i; }
        } else {
            n.t3 = s;
        }
    }
}
__device__ __forceinline__ void near_merge(NearTop &n, const NearTop &o)
{
    near_insert(n, o.t1, o.i1);
    near_insert(n, o.t2, o.i2);
    if (o.t3 < n.t3) n.t3 = o.t3;        // not below n.t2: o.t2 has been inserted
}
// How far above the smallest lower bound (of a centre with squared norm nc) a rival's may lie.
template <bool kHalf>
__device__ __forceinline__ float near_slack(float nx, float nc)
{
    return 2.f * kNearErr * (nx + nc) + (kHalf ? 1.4e-6f * sqrtf(nx) : 0.f) + 1e-34f;
}

// A centre component as hi + mid. A centre with components beyond the element type, or whose squared norm fp32 cannot
// hold, is stored as zeros with a bound of -inf: it is a candidate of every point.
template <bool kHalf>
__device__ __forceinline__ void split_component(double v, uint16_t &hi, uint16_t &mid)
{
    hi = double_to_elem<kHalf>(v);
    mid = double_to_elem<kHalf>(v - elem_to_double<kHalf>(hi));
}
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
    uint4 ring[2][2][kNearTile * 16];    // [stage][hi, mid]: 64 rows of 256 bytes, 16-byte pieces XOR-swizzled
    float bias[2][kNearTile];
    float largest;                       // largest squared norm among the centres (fp32 source only)
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
    uint4 *rows = &sm.ring[0][0][0];                        // 64 KB: the whole ring
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
    NearTop top[4];                                         // rows g, g + 8, g + 16, g + 24 of the warp's 32
#pragma unroll
    for (int r = 0; r < 4; ++r) top[r] = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, k_lo, k_lo};
    fill(0, k_lo, min(kNearTile, k_hi - k_lo));
    asm volatile("cp.async.commit_group;");
    int stage = 0;
    for (int base = k_lo; base < k_hi; base += kNearTile, stage ^= 1) {
        if (base + kNearTile < k_hi) fill(stage ^ 1, base + kNearTile, min(kNearTile, k_hi - base - kNearTile));
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const uint32_t hi_a = shared_addr(&sm.ring[stage][0][0]), mid_a = shared_addr(&sm.ring[stage][1][0]);
#pragma unroll 2
        for (int nt = 0; nt < kNearTile / 8; ++nt) {
            const int row = nt * 8 + (lane & 7);
            float ah[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, am[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) {
                uint32_t bh[4], bm[4];
                const uint32_t at = (uint32_t)near_piece(row, 4 * s2 + (lane >> 3)) * 16u;
                ldmatrix4(bh, hi_a + at);
                ldmatrix4(bm, mid_a + at);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint32_t(&f)[4] = a[m][2 * s2 + h];
                        mma_rows<kHalf>(ah[m], f[0], f[1], f[2], f[3], bh[2 * h], bh[2 * h + 1]);
                        mma_rows<kHalf>(am[m], f[0], f[1], f[2], f[3], bm[2 * h], bm[2 * h + 1]);
                    }
            }
            const float2 bias = *reinterpret_cast<const float2 *>(&sm.bias[stage][nt * 8 + 2 * c]);
            const int col = base + nt * 8 + 2 * c;
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    near_insert(top[2 * m + (e >> 1)], fmaf(-2.f, ah[m][e] + am[m][e], (e & 1) ? bias.y : bias.x), col + (e & 1));
        }
        __syncthreads();                                    // the stage may be filled again
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            NearTop n;
            n.t1 = __shfl_xor_sync(0xFFFFFFFFu, top[r].t1, o);
            n.t2 = __shfl_xor_sync(0xFFFFFFFFu, top[r].t2, o);
            n.t3 = __shfl_xor_sync(0xFFFFFFFFu, top[r].t3, o);
            n.i1 = __shfl_xor_sync(0xFFFFFFFFu, top[r].i1, o);
            n.i2 = __shfl_xor_sync(0xFFFFFFFFu, top[r].i2, o);
            near_merge(top[r], n);
        }
        if (c == 0) sm.top[warp * 32 + 8 * r + (lane >> 2)] = top[r];
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
