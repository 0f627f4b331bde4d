// Algorithm 2 on the rows of one parent held in shared memory: representatives, owners, packed order.
//
// The records are defined by fp64 distances summed over the dimensions in increasing order (multiply and
// add rounded separately), with the paper's index tie rules. Those sums are only needed where they
// decide something: every comparison is first made on fp32 distances |x|^2 + |y|^2 - 2 x.y whose dot products
// come from tensor cores, with a bound on their error, and a comparison that the bound leaves open is
// made again on the fp64 sums. The result is the fp64 one as long as the bound holds.
//
// The bound. With S = sum |x_d y_d| <= B, B = the largest squared norm in the parent: products of two 16-bit
// values are exact in fp32; an MMA over 16 of them adds 17 terms, each with an error of at most 2^-23 of the
// magnitudes summed so far; at most 8 MMAs follow one another in an accumulator (longer rows start a new
// one and add it to an fp32 total). That error per term is an assumption: order and rounding of the sum inside
// an MMA are not specified. Measured over 128 values, six distributions (cancelling, all positive, sorted by size ...),
// mma.sync and tcgen05: at most 13 * 2^-23 of S where the bound has 136. That is 8 * 17 * 2^-23 * B for a dot product and four times that,
// plus the rounding of the last few operations, for a distance: 2^-13.85 B. kDistErr is 5 % above. A score
// against the parent's mean (norm minus twice the mean of the row's dot products) has a smaller
// error. The fp64 sums are within 2^-44 of the true values, which the 5 % covers as well. A product below the range of
// normal fp32 numbers may lose up to 2^-126 whatever the size of its factors; a distance has at most 4 * 576 such
// losses, 3e-35, and kUnderflow stands for them in every bound that is relative to the two rows at hand. Where fp32
// could overflow or loses most products (B outside [1e-30, 1e37], or not a number) the bound is infinite:
// then every comparison is made on the fp64 sums.
#pragma once
#include <limits.h>
#include <math_constants.h>

#include "common.cuh"

namespace santapp {

constexpr float kDistErr = 7.2e-5f;      // error bound of an fp32 distance, in units of the largest squared norm
constexpr float kUnderflow = 1e-34f;     // and in absolute terms: products and squares that fp32 holds as subnormals or loses

template <bool kHalf>
__device__ __forceinline__ void mma_rows(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    if constexpr (kHalf)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                     : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                     : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t shared_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void copy16_async(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ float dist_error(float largest_norm)
{
    return largest_norm >= 1e-30f && largest_norm <= 1e37f ? fmaf(kDistErr, largest_norm, kUnderflow) : CUDART_INF_F;
}
__device__ __forceinline__ float norm_or_inf(float n) { return n <= 1e37f ? n : CUDART_INF_F; }

// Rows of 256 bytes in shared memory, 16-byte pieces XOR-swizzled: ldmatrix without bank conflicts.
__device__ __forceinline__ int near_piece(int row, int chunk) { return row * 16 + (chunk ^ (row & 7)); }

// The defining distance of two rows (words of two 16-bit values each); not a number counts as infinitely far.
template <bool kHalf>
__device__ __forceinline__ double exact_dist(const uint32_t *a, const uint32_t *b, int n_words)
{
    double s = 0.0;
#pragma unroll 8
    for (int w = 0; w < n_words; ++w) {
        const uint32_t x = a[w], y = b[w];
        const double e0 = __dsub_rn((double)elem_lo<kHalf>(x), (double)elem_lo<kHalf>(y));
        const double e1 = __dsub_rn((double)elem_hi<kHalf>(x), (double)elem_hi<kHalf>(y));
        s = __dadd_rn(s, __dmul_rn(e0, e0));
        s = __dadd_rn(s, __dmul_rn(e1, e1));
    }
    return s == s ? s : CUDART_INF;
}

// Warp-wide arg-min / arg-max over the lanes in `mask` (ties to the smaller index); every lane gets the index.
template <bool kMin>
__device__ __forceinline__ int warp_arg(double v, int i, bool in)
{
    if (!in) { v = kMin ? CUDART_INF : -CUDART_INF; i = INT_MAX; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        const int j = __shfl_xor_sync(0xFFFFFFFFu, i, o);
        const bool take = (kMin ? w < v : w > v) || (w == v && j < i);
        if (take) { v = w; i = j; }
    }
    return i;
}
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// A parent of at most kRows <= 32 rows, one warp, lane i = row i. rows: kRows rows of kPitch words in shared
// memory (kPitch * 4 an odd multiple of 16 bytes: ldmatrix without bank conflicts), of which the first kWords
// take part in distances; what lies in the rows past nC is never looked at. dist: [kRows][kRows + 1] floats of
// scratch. All distances of the parent come out of one product of the rows with themselves (the fragment of
// 16 rows as the first operand is also the fragment of its two groups of 8 rows as the second).
// Results: `owner` of the lane's row, rep_of[u] in shared memory, and the position of the row in packed order.
template <int kRows, int kWords, int kPitch, bool kHalf>
__device__ __forceinline__ void select_small(const uint32_t *rows, float *dist, int *rep_of, int nC, int r, int &owner_out, int &pos_out)
{
    constexpr int kTiles = kRows / 16, kGroups = kRows / 8, kDp = kRows + 1;
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    {
        float tot[kTiles][kGroups][4];
#pragma unroll
        for (int m = 0; m < kTiles; ++m)
#pragma unroll
            for (int n = 0; n < kGroups; ++n) tot[m][n][0] = tot[m][n][1] = tot[m][n][2] = tot[m][n][3] = 0.f;
        // lane l addresses row (l & 7) + 8 * bit 3 of l, 16-byte piece bit 4 of l
        const uint32_t base = shared_addr(rows) + (uint32_t)((lane & 15) * kPitch * 4 + (lane >> 4) * 16);
#pragma unroll 1
        for (int part = 0; part < kWords / 64; ++part) {             // 8 MMAs of 16 values each
            float acc[kTiles][kGroups][4];
#pragma unroll
            for (int m = 0; m < kTiles; ++m)
#pragma unroll
                for (int n = 0; n < kGroups; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                uint32_t a[kTiles][4];
#pragma unroll
                for (int m = 0; m < kTiles; ++m) ldmatrix4(a[m], base + (uint32_t)(m * 16 * kPitch * 4 + (part * 8 + k) * 32));
#pragma unroll
                for (int m = 0; m < kTiles; ++m)
#pragma unroll
                    for (int n = 0; n < kGroups; ++n)
                        mma_rows<kHalf>(acc[m][n], a[m][0], a[m][1], a[m][2], a[m][3], a[n >> 1][n & 1], a[n >> 1][2 + (n & 1)]);
            }
#pragma unroll
            for (int m = 0; m < kTiles; ++m)
#pragma unroll
                for (int n = 0; n < kGroups; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) tot[m][n][e] += acc[m][n][e];
        }
#pragma unroll
        for (int m = 0; m < kTiles; ++m)
#pragma unroll
            for (int n = 0; n < kGroups; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) dist[(16 * m + g + 8 * (e >> 1)) * kDp + 8 * n + 2 * c + (e & 1)] = tot[m][n][e];
    }
    __syncwarp();
    const bool live = lane < nC;
    const int me = live ? lane : 0;
    const float norm = dist[me * kDp + me];
    const float err = dist_error(warp_max(norm_or_inf(norm)));
    const uint32_t *my_row = rows + me * kPitch;

    // first representative: the row nearest the mean. |x - mu|^2 less |mu|^2, from the row's dot products
    int rep;
    {
        float sum = 0.f;
        for (int j = 0; j < nC; ++j) sum += dist[me * kDp + j];
        const float score = norm - 2.f * sum / (float)nC;
        const float best = -warp_max(live ? -score : -CUDART_INF_F);
        const bool maybe = live && !(score > best + 2.f * err);
        const unsigned who = __ballot_sync(0xFFFFFFFFu, maybe);
        if (__popc(who) == 1) {
            rep = __ffs(who) - 1;
        } else {
            // the mean in fp64 (rows in token order, one division), 32 dimensions at a time, one per lane
            double s = 0.0;
#pragma unroll 1
            for (int d0 = 0; d0 < 2 * kWords; d0 += 32) {
                double mu = 0.0;
                for (int i = 0; i < nC; ++i) {
                    const uint32_t w = rows[i * kPitch + (d0 + lane) / 2];
                    mu = __dadd_rn(mu, (double)((lane & 1) ? elem_hi<kHalf>(w) : elem_lo<kHalf>(w)));
                }
                mu = __ddiv_rn(mu, (double)nC);
#pragma unroll 4
                for (int t = 0; t < 32; ++t) {
                    const double m = __shfl_sync(0xFFFFFFFFu, mu, t);
                    const uint32_t w = my_row[(d0 + t) / 2];
                    const double e = __dsub_rn((double)((t & 1) ? elem_hi<kHalf>(w) : elem_lo<kHalf>(w)), m);
                    s = __dadd_rn(s, __dmul_rn(e, e));
                }
            }
            rep = min(warp_arg<true>(s == s ? s : CUDART_INF, lane, maybe), nC - 1);
        }
    }

    // farthest-first representatives; the running (nearest distance, owner) pair is the nearest-
    // representative assignment with ties going to the earlier-selected one
    float mind = CUDART_INF_F;
    int owner = 0;
    bool is_rep = false;
    double near = 0.0;                                            // the fp64 distance to the owner, once a comparison needed it
    bool known = false;
    for (int u = 0; u < r; ++u) {
        if (lane == 0) rep_of[u] = rep;
        is_rep |= lane == rep;
        __syncwarp();
        const float nr = dist[rep * kDp + rep];
        const float d = lane == rep ? 0.f : norm + nr - 2.f * dist[me * kDp + rep];
        bool closer = u == 0 || d < mind - 2.f * err;
        const bool open = live && u > 0 && !closer && !(d > mind + 2.f * err) && !(known && near == 0.0);      // (nothing is nearer than zero)
        if (open) {
            const double d_new = exact_dist<kHalf>(my_row, rows + rep * kPitch, kWords);
            if (!known) near = exact_dist<kHalf>(my_row, rows + rep_of[owner] * kPitch, kWords);
            closer = d_new < near;
            if (closer) near = d_new;
        }
        known = open || (known && !closer);
        if (closer) owner = u;
        mind = open ? fminf(mind, d) : (closer ? d : mind);       // either value is within the bound of the smaller one
        if (u + 1 < r) {
            const bool can = live && !is_rep;
            const float far = warp_max(can ? mind : -CUDART_INF_F);
            const bool maybe = can && !(mind < far - 2.f * err);
            const unsigned who = __ballot_sync(0xFFFFFFFFu, maybe);
            if (__popc(who) == 1) {
                rep = __ffs(who) - 1;
            } else {
                if (maybe && !known) near = exact_dist<kHalf>(my_row, rows + rep_of[owner] * kPitch, kWords);
                known |= maybe;
                rep = min(warp_arg<false>(near, lane, maybe), nC - 1);
            }
        }
    }
    for (int u = 0; u < r; ++u)                                   // a representative owns its own row
        if (rep_of[u] == lane) owner = u;
    // packed order: teams in selection order, members by index
    int pos = 0;
    for (int j = 0; j < nC; ++j) {
        const int o = __shfl_sync(0xFFFFFFFFu, owner, j);
        pos += (o < owner || (o == owner && j < lane)) ? 1 : 0;
    }
    owner_out = owner;
    pos_out = pos;
}

}  // namespace santapp
