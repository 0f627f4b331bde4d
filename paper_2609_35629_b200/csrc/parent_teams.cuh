// Records of one parent (Algorithm 2 and the packed copy), by a warp for at most 32 rows and by a block for 33 to 512:
// used by the contiguous builder (parents are ranges of tokens) and by the builder on a given partition (parents
// are member lists). select_rows.cuh says how the teams are found without evaluating most fp64 distances.
#pragma once
#include <limits.h>

#include "build_util.cuh"
#include "common.cuh"
#include "select_rows.cuh"

namespace santapp {
namespace {

constexpr int kPitch = 68;               // words per staged key: 64 of data and 4 of padding (ldmatrix without bank conflicts)
constexpr int kWords = 64;

// A parent and where its records go. Its rows occupy [s0, s0 + nC) of the sequence's packed order: teams are numbered
// parent by parent, so nothing outside the parent decides where its rows go.
struct ParentRows {
    const uint16_t *k_prompt, *v_prompt;
    uint16_t *k_packed, *v_packed, *rep_keys;
    int32_t *row_token;
    size_t plane;                        // first row of the sequence in a [n_kv][rows_total] array
    int s0, nC, r;                       // first packed row, rows, teams
    const int32_t *members;              // tokens of the rows, or null: tokens s0, s0 + 1, ...
    int32_t *csr;                        // row offset of the parent's first team
    size_t rep0;                         // the parent's first representative in [n_kv][teams_total]
    float *abs_max;                      // of the pair, zero before the kernel
};

// The largest magnitude (bits of a 16-bit value) as the pair's bound on |representative key|; the array is zero
// before the kernel runs, and non-negative floats order like their bits.
template <bool kHalf>
__device__ __forceinline__ void raise_abs_max(float *dst, uint32_t m)
{
    const float v = kHalf ? elem_to_float<true>((uint16_t)m) : __uint_as_float(m << 16);
    atomicMax(reinterpret_cast<uint32_t *>(dst), __float_as_uint(v));
}
__device__ __forceinline__ uint32_t magnitude2(uint32_t w) { return max(w & 0x7FFFu, (w >> 16) & 0x7FFFu); }

// ---- at most 32 rows: one warp ----
// Bound by memory (K and V read once and written once, 1 KB of each row), as long as enough rows are on their
// way: a warp has its parent's K in flight as asynchronous copies and its V in registers before it
// computes anything, 8 to 16 KB, and about 20 warps are resident.
template <int kRows>
struct SmallSmem {
    __align__(16) uint32_t rows[kRows * kPitch];
    float dist[kRows * (kRows + 1)];
    int rep_of[32];
};
template <int kRows, bool kHalf>
__device__ __forceinline__ void small_parent(const ParentRows &t, SmallSmem<kRows> &sm)
{
    const int lane = threadIdx.x & 31, q = lane & 15;
    const int token = t.members ? t.members[min(lane, t.nC - 1)] : t.s0 + lane;
    const uint4 *k = reinterpret_cast<const uint4 *>(t.k_prompt) + t.plane * 16;
    const uint4 *v = reinterpret_cast<const uint4 *>(t.v_prompt) + t.plane * 16;
    uint4 vr[kRows / 2];
#pragma unroll
    for (int m = 0; m < kRows / 2; ++m) {                    // a row per half warp
        const int i = 2 * m + (lane >> 4);
        const size_t at = (size_t)__shfl_sync(0xFFFFFFFFu, token, i) * 16 + q;
        if (i < t.nC) copy16_async(shared_addr(sm.rows + i * kPitch + q * 4), k + at);
        vr[m] = i < t.nC ? __ldg(v + at) : make_uint4(0u, 0u, 0u, 0u);
    }
    copy_async_wait();
    __syncwarp();
    int owner, pos;
    select_small<kRows, kWords, kPitch, kHalf>(sm.rows, sm.dist, sm.rep_of, t.nC, t.r, owner, pos);
    uint4 *kdst = reinterpret_cast<uint4 *>(t.k_packed) + (t.plane + t.s0) * 16;
    uint4 *vdst = reinterpret_cast<uint4 *>(t.v_packed) + (t.plane + t.s0) * 16;
#pragma unroll
    for (int m = 0; m < kRows / 2; ++m) {
        const int i = 2 * m + (lane >> 4);
        const int d = __shfl_sync(0xFFFFFFFFu, pos, i);
        if (i < t.nC) {
            kdst[d * 16 + q] = *reinterpret_cast<const uint4 *>(sm.rows + i * kPitch + q * 4);
            vdst[d * 16 + q] = vr[m];
        }
    }
    if (lane < t.nC) t.row_token[t.plane + t.s0 + pos] = token;
    int upto = 0;                                           // rows of the teams 0 .. lane
    for (int i = 0; i < t.nC; ++i) upto += __shfl_sync(0xFFFFFFFFu, owner, i) <= lane ? 1 : 0;
    if (lane < t.r) t.csr[1 + lane] = t.s0 + upto;
    uint32_t m = 0u;
    uint4 *rdst = reinterpret_cast<uint4 *>(t.rep_keys) + t.rep0 * 16;
    for (int e = lane; e < t.r * 16; e += 32) {
        const uint4 w = *reinterpret_cast<const uint4 *>(sm.rows + sm.rep_of[e >> 4] * kPitch + (e & 15) * 4);
        rdst[e] = w;
        m = max(m, max(max(magnitude2(w.x), magnitude2(w.y)), max(magnitude2(w.z), magnitude2(w.w))));
    }
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0) raise_abs_max<kHalf>(t.abs_max, m);
}

// ---- 33 to 512 rows: one block ----
// Farthest-first selection is a chain of R dependent steps. A step here costs one block barrier: the distances
// to the next representative are already in shared memory. They come from products of all rows with
// eight candidate rows at a time (an MMA's eight columns): the representative just chosen and the rows that
// are farthest now, which are the ones chosen next unless a new representative happens to lie near
// them; when a choice is not among the candidates, the next eight are multiplied (about six times for 32
// representatives of 512 rows). A warp's rows stay in its registers as MMA operands for that.
// 512 rows are one block per SM (131 KB of keys): 8 warps with two rows per thread rather than 16 with one,
// since the step is a chain of warp-wide reductions and a barrier, which fewer warps finish sooner.
struct LargeTop {                        // a warp's farthest row: bounds of its distance, the largest upper bound of
    float lo, hi, hi_others;             //   the warp's other rows, and its index
    int row;
};
// Up to 256 rows as many blocks share an SM as make sixteen warps: with a block or two, whatever registers the compiler takes
// when it is not told (199 for 64 to 256 rows, where 125 do without spills), the chain of one block has nothing beside it.
// 4 x 32K keys in parents of 256 / 128 / 64: 82 -> 60, 57 -> 44, 59 -> 44 us.
__host__ __device__ constexpr int large_blocks(int warps, int rows_per_thread) { return rows_per_thread > 1 ? 1 : 16 / warps; }
template <int kWarps, int kRpt>
struct LargeSmem {
    static constexpr int kT = 32 * kWarps, kRows = kT * kRpt; // threads, rows
    static constexpr int kDistPitch = kRows + 4;              // floats per candidate: conflict-free fragment stores
    uint32_t rows[kRows * kPitch];
    union {
        float dist[8][kDistPitch];                            // fp32 squared distances to the candidates
        uint16_t count[kWarps * kRpt][kRows];                 // rows of each team in each group of 32 rows, then their prefix
    };
    float norm[kRows];
    double mu64[kHeadDim];
    double near[kRows];                                       // fp64 distances to the owners, of the rows that a choice needed them of
    float mu[4][kHeadDim];
    LargeTop top[2][kWarps];
    uint32_t next_key[2 * kWarps];                            // two rows of each warp for the next candidates
    int next_row[2 * kWarps];
    int cand[kWarps][8];
    float red[3][kWarps];
    uint16_t rep_of[kRows];
    uint16_t owner[kRows];
    int team_start[kRows];
    int token[kRows];
    ValIdx arg[33];
    int scan[33];
};
#define LARGE_ROW(k) (warp * 32 * kRpt + 32 * (k) + lane)     // the thread's k-th row

// The row nearest the mean among those with a bit in `maybe` (bit k: the thread's k-th row), by the defining fp64
// sums (mean: rows in token order, one division; ties to the smaller index). Whole block.
template <int kWarps, int kRpt, bool kHalf>
__device__ __noinline__ int nearest_mean_exact(LargeSmem<kWarps, kRpt> &sm, int nC, unsigned maybe)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
    for (int d = tid; d < kHeadDim; d += 32 * kWarps) {
        double s = 0.0;
#pragma unroll 8
        for (int i = 0; i < nC; ++i) {
            const uint32_t w = sm.rows[i * kPitch + (d >> 1)];
            s = __dadd_rn(s, (double)((d & 1) ? elem_hi<kHalf>(w) : elem_lo<kHalf>(w)));
        }
        sm.mu64[d] = __ddiv_rn(s, (double)nC);
    }
    __syncthreads();
    ValIdx best = {CUDART_INF, INT_MAX};
    for (int k = 0; k < kRpt; ++k) {
        if (!((maybe >> k) & 1u)) continue;
        const uint32_t *row = sm.rows + LARGE_ROW(k) * kPitch;
        double s = 0.0;
#pragma unroll 4
        for (int w = 0; w < kWords; ++w) {
            const uint32_t word = row[w];
            const double e0 = __dsub_rn((double)elem_lo<kHalf>(word), sm.mu64[2 * w]);
            const double e1 = __dsub_rn((double)elem_hi<kHalf>(word), sm.mu64[2 * w + 1]);
            s = __dadd_rn(s, __dmul_rn(e0, e0));
            s = __dadd_rn(s, __dmul_rn(e1, e1));
        }
        best = pick<true>(best, {s == s ? s : CUDART_INF, LARGE_ROW(k)});
    }
    best = block_arg<true>(best, sm.arg);
    return min(best.i, nC - 1);
}

// The defining fp64 evaluation of a parent by a block, for parents on which the fp32 distances decide too
// little (rows that repeat many times, values outside the range of the error bound).
template <int kWarps, int kRpt, bool kHalf>
__device__ __noinline__ void select_large_exact(LargeSmem<kWarps, kRpt> &sm, int nC, int r)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned live = 0u, is_rep = 0u;
    double mind[kRpt];
    int owner[kRpt];
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        live |= (LARGE_ROW(k) < nC ? 1u : 0u) << k;
        mind[k] = CUDART_INF;
        owner[k] = 0;
    }
    int rep = nearest_mean_exact<kWarps, kRpt, kHalf>(sm, nC, live);
    for (int u = 0; u < r; ++u) {
        if (tid == 0) sm.rep_of[u] = (uint16_t)rep;
        ValIdx far = {-2.0, INT_MAX};
#pragma unroll
        for (int k = 0; k < kRpt; ++k) {
            if (!((live >> k) & 1u)) continue;
            if (LARGE_ROW(k) == rep) is_rep |= 1u << k;
            const double d = exact_dist<kHalf>(sm.rows + LARGE_ROW(k) * kPitch, sm.rows + rep * kPitch, kWords);
            if (d < mind[k]) { mind[k] = d; owner[k] = u; }
            far = pick<false>(far, {((is_rep >> k) & 1u) ? -1.0 : mind[k], LARGE_ROW(k)});
        }
        if (u + 1 < r) rep = min(block_arg<false>(far, sm.arg).i, nC - 1);
    }
#pragma unroll
    for (int k = 0; k < kRpt; ++k) sm.owner[LARGE_ROW(k)] = (uint16_t)owner[k];
    __syncthreads();
}

// What a parent's open comparisons may cost before it goes to the fp64 evaluation, which starts over: half of what
// that takes. Unit: a warp's fp64 distances to one representative, of which the evaluation makes r for every 32 rows;
// an open row takes one per 32 representatives, a choice among rows whose distances are known about kChoiceCost.
constexpr int kChoiceCost = 1;

// The first of a row's nearest representatives among the first n, by the defining distances: a warp, whose lanes take the
// representatives. Every lane gets it and the distance.
template <bool kHalf, int kWarps, int kRpt>
__device__ __forceinline__ int nearest_rep(const LargeSmem<kWarps, kRpt> &sm, int i, int n, double &dist)
{
    const int lane = threadIdx.x & 31;
    double near = CUDART_INF;
    int who = INT_MAX;
    for (int q = lane; q < n; q += 32) {
        const double d = exact_dist<kHalf>(sm.rows + i * kPitch, sm.rows + sm.rep_of[q] * kPitch, kWords);
        if (d < near || who == INT_MAX) { near = d; who = q; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double d = __shfl_xor_sync(0xFFFFFFFFu, near, o);
        const int w = __shfl_xor_sync(0xFFFFFFFFu, who, o);
        if (d < near || (d == near && w < who)) { near = d; who = w; }
    }
    dist = near;
    return who;
}

template <int kWarps, int kRpt, bool kHalf>
__device__ __forceinline__ void select_large(LargeSmem<kWarps, kRpt> &sm, int nC, int r)
{
    constexpr int kT = 32 * kWarps;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, c = lane & 3;
    // the mean, approximately (fp32 sums), then every row's norm and its distance to the mean
    constexpr int kParts = kT / kWords;
    static_assert(kParts >= 1 && kParts <= 4 && kParts * 128 >= LargeSmem<kWarps, kRpt>::kRows, "a word per thread; chains of at most 128 additions");
    {
        const int word = tid & (kWords - 1), part = tid / kWords;
        float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
        for (int i = part; i < nC; i += kParts) {
            const uint32_t w = sm.rows[i * kPitch + word];
            s0 += elem_lo<kHalf>(w);
            s1 += elem_hi<kHalf>(w);
        }
        sm.mu[part][2 * word] = s0;
        sm.mu[part][2 * word + 1] = s1;
    }
    __syncthreads();
    for (int d = tid; d < kHeadDim; d += kT) {
        float s = sm.mu[0][d];
#pragma unroll
        for (int q = 1; q < kParts; ++q) s += sm.mu[q][d];
        sm.mu[0][d] = s / (float)nC;
    }
    __syncthreads();
    unsigned live = 0u, is_rep = 0u;
    float norm[kRpt], mind[kRpt], lo[kRpt], hi[kRpt];         // squared norm; nearest distance and its bounds
    float sum_norm = 0.f, largest = 0.f;
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        const int i = LARGE_ROW(k);
        live |= (i < nC ? 1u : 0u) << k;
        norm[k] = mind[k] = 0.f;
    }
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
        const float4 m0 = *reinterpret_cast<const float4 *>(&sm.mu[0][8 * q]), m1 = *reinterpret_cast<const float4 *>(&sm.mu[0][8 * q + 4]);
        const float m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
        for (int k = 0; k < kRpt; ++k) {
            const uint4 w4 = *reinterpret_cast<const uint4 *>(sm.rows + (LARGE_ROW(k) < nC ? LARGE_ROW(k) : 0) * kPitch + 4 * q);
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const float x0 = elem_lo<kHalf>(w[t]), x1 = elem_hi<kHalf>(w[t]);
                const float e0 = x0 - m[2 * t], e1 = x1 - m[2 * t + 1];
                norm[k] = fmaf(x0, x0, norm[k]);
                norm[k] = fmaf(x1, x1, norm[k]);
                mind[k] = fmaf(e0, e0, mind[k]);
                mind[k] = fmaf(e1, e1, mind[k]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        sm.norm[LARGE_ROW(k)] = norm[k];
        largest = fmaxf(largest, norm_or_inf(norm[k]));
        sum_norm += ((live >> k) & 1u) ? norm[k] : 0.f;
    }
    largest = warp_max(largest);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum_norm += __shfl_xor_sync(0xFFFFFFFFu, sum_norm, o);
    if (lane == 0) { sm.red[0][warp] = largest; sm.red[1][warp] = sum_norm; }
    __syncthreads();
    sum_norm = largest = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { largest = fmaxf(largest, sm.red[0][w]); sum_norm += sm.red[1][w]; }
    if (!(dist_error(largest) < CUDART_INF_F)) { select_large_exact<kWarps, kRpt, kHalf>(sm, nC, r); return; }
    // First representative: the row nearest the mean. With A the mean length of the rows, the fp32 mean is
    // within 131 * 2^-24 A of the fp64 one (chains of 128 additions), and the distance to it within
    // 2 (|x| + A) * 131 * 2^-24 A + 2^-17 (|x| + A)^2 <= 4.8e-5 (|x|^2 + A^2); A^2 is at most the mean squared norm.
    const float mean_norm = sum_norm / (float)nC;
    float best = CUDART_INF_F;
#pragma unroll
    for (int k = 0; k < kRpt; ++k)
        if ((live >> k) & 1u) best = fminf(best, mind[k] + fmaf(kDistErr, norm[k] + mean_norm, kUnderflow));
    best = -warp_max(-best);
    if (lane == 0) sm.red[2][warp] = best;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) best = fminf(best, sm.red[2][w]);
    unsigned maybe = 0u;
#pragma unroll
    for (int k = 0; k < kRpt; ++k)
        if (((live >> k) & 1u) && !(mind[k] - fmaf(kDistErr, norm[k] + mean_norm, kUnderflow) > best)) { maybe |= 1u << k; sm.rep_of[0] = (uint16_t)LARGE_ROW(k); }
    const bool one = __syncthreads_count(maybe != 0u) == 1 && __syncthreads_count(__popc(maybe) > 1) == 0;
    int rep = one ? sm.rep_of[0] : nearest_mean_exact<kWarps, kRpt, kHalf>(sm, nC, maybe);

    // the warp's rows as MMA operands
    const uint32_t rows_a = shared_addr(sm.rows);
    uint32_t a[2 * kRpt][8][4];
#pragma unroll
    for (int m = 0; m < 2 * kRpt; ++m)
#pragma unroll
        for (int s = 0; s < 8; ++s)
            ldmatrix4(a[m][s], rows_a + (uint32_t)((warp * 32 * kRpt + 16 * m + (lane & 15)) * kPitch * 4 + (lane >> 4) * 16 + s * 32));

    constexpr float kPairErr = 0.5f * kDistErr;               // times the sum of the two squared norms, plus kUnderflow
    const int budget = max(16, r * kRpt * kWarps / 2);
    int owner[kRpt], parity = 0, u = 0, spent = 0;
    unsigned open_owner = 0u;                                 // bit k: the bound leaves the nearest representative open
    unsigned known = 0u;                                      // bit k: sm.near holds the row's distance
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        owner[k] = 0;
        if (LARGE_ROW(k) == rep) is_rep |= 1u << k;
        lo[k] = hi[k] = mind[k];                              // until the first distances are there: who is far from the mean
    }
    while (true) {
        // ---- the next eight candidates: `rep`, and the seven farthest of two rows of every warp ----
        {
            uint32_t key = 0u, key2 = 0u;                     // the thread's farthest row that is not a representative, and its next
            int row = -1, row2 = -1;
#pragma unroll
            for (int k = 0; k < kRpt; ++k) {
                const uint32_t v = ((live & ~is_rep) >> k) & 1u ? __float_as_uint(mind[k]) + 1u : 0u;
                if (v > key) { key2 = key; row2 = row; key = v; row = LARGE_ROW(k); }
                else if (v > key2) { key2 = v; row2 = LARGE_ROW(k); }
            }
            const uint32_t k0 = __reduce_max_sync(0xFFFFFFFFu, key);
            const int l0 = __ffs(__ballot_sync(0xFFFFFFFFu, key == k0)) - 1;
            const uint32_t rest = lane == l0 ? key2 : key;
            const int rest_row = lane == l0 ? row2 : row;
            const uint32_t k1 = __reduce_max_sync(0xFFFFFFFFu, rest);
            const int l1 = __ffs(__ballot_sync(0xFFFFFFFFu, rest == k1)) - 1;
            if (lane == l0) { sm.next_key[2 * warp] = k0; sm.next_row[2 * warp] = row; }
            if (lane == l1) { sm.next_key[2 * warp + 1] = k1; sm.next_row[2 * warp + 1] = rest_row; }
        }
        __syncthreads();
        {
            constexpr int kTops = 2 * kWarps;                 // at most 16
            const uint32_t key = lane < kTops ? sm.next_key[lane] : 0u;
            if (lane < 8) sm.cand[warp][lane] = rep;
            int rank = 0;
#pragma unroll
            for (int o = 0; o < kTops; ++o) {
                const uint32_t k = sm.next_key[o];
                rank += (k > key || (k == key && o < lane)) ? 1 : 0;
            }
            __syncwarp();
            if (key != 0u && rank < 7) sm.cand[warp][rank + 1] = sm.next_row[lane];
            __syncwarp();
        }
        const int cand = lane < 8 ? sm.cand[warp][lane] : -1;
        // ---- distances of the warp's rows to them ----
        {
            const uint32_t b_addr = rows_a + (uint32_t)(sm.cand[warp][lane & 7] * kPitch * 4 + (lane >> 3) * 16);
            float acc[2 * kRpt][4];
#pragma unroll
            for (int m = 0; m < 2 * kRpt; ++m) acc[m][0] = acc[m][1] = acc[m][2] = acc[m][3] = 0.f;
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) {
                uint32_t bf[4];
                ldmatrix4(bf, b_addr + s2 * 64);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int m = 0; m < 2 * kRpt; ++m) {
                        const uint32_t(&f)[4] = a[m][2 * s2 + h];
                        mma_rows<kHalf>(acc[m], f[0], f[1], f[2], f[3], bf[2 * h], bf[2 * h + 1]);
                    }
            }
            const float n0 = sm.norm[sm.cand[warp][2 * c]], n1 = sm.norm[sm.cand[warp][2 * c + 1]];
            // (a warp reads only its own rows' distances: no block barrier)
#pragma unroll
            for (int m = 0; m < 2 * kRpt; ++m)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = warp * 32 * kRpt + 16 * m + g + 8 * (e >> 1);
                    const float d = sm.norm[i] + ((e & 1) ? n1 : n0) - 2.f * acc[m][e];
                    sm.dist[2 * c + (e & 1)][i] = fmaxf(d, 0.f);
                }
        }
        __syncwarp();
        // ---- selection steps as long as the choice is among the candidates ----
        int col = 0;
        bool done = false;
        while (true) {
            if (tid == 0) sm.rep_of[u] = (uint16_t)rep;
            const float rep_norm = sm.norm[rep];
            float top_lo = -1.f, top_hi = -1.f, others = -1.f;
            int top_row = 0;
#pragma unroll
            for (int k = 0; k < kRpt; ++k) {
                const float d = sm.dist[col][LARGE_ROW(k)], e = fmaf(kPairErr, norm[k] + rep_norm, kUnderflow);
                if (u == 0 || d + e < lo[k]) {                // certainly nearer than every earlier one
                    mind[k] = d; lo[k] = d - e; hi[k] = d + e; owner[k] = u;
                    open_owner &= ~(1u << k);
                    known &= ~(1u << k);
                } else if (!(d - e > hi[k]) && hi[k] > 0.f) { // not certain: the minimum lies between the smaller bounds
                    if (d < mind[k]) { mind[k] = d; owner[k] = u; }
                    lo[k] = fminf(lo[k], d - e);
                    hi[k] = fminf(hi[k], d + e);
                    open_owner |= 1u << k;
                    known &= ~(1u << k);
                }
                if (((live & ~is_rep) >> k) & 1u) {
                    if (lo[k] > top_lo || top_row == 0) {
                        others = fmaxf(others, top_hi);
                        top_lo = fmaxf(lo[k], 0.f); top_hi = hi[k]; top_row = LARGE_ROW(k) + 1;
                    } else {
                        others = fmaxf(others, hi[k]);
                    }
                }
            }
            ++u;
            if (u == r) { done = true; break; }
            {
                // the warp's row with the largest lower bound; the others by their upper bounds
                const uint32_t key = top_row ? __float_as_uint(top_lo) + 1u : 0u;
                const uint32_t k0 = __reduce_max_sync(0xFFFFFFFFu, key);
                const int l0 = __ffs(__ballot_sync(0xFFFFFFFFu, key == k0)) - 1;
                const float rest = lane == l0 ? others : fmaxf(others, top_hi);
                const uint32_t k1 = __reduce_max_sync(0xFFFFFFFFu, rest >= 0.f ? __float_as_uint(rest) + 1u : 0u);
                if (lane == l0)
                    sm.top[parity][warp] = {k0 ? top_lo : -1.f, k0 ? top_hi : -1.f, k1 ? __uint_as_float(k1 - 1u) : -1.f, top_row - 1};
            }
            __syncthreads();
            const LargeTop t = sm.top[parity][min(lane, kWarps - 1)];
            parity ^= 1;
            const uint32_t key = lane < kWarps && t.lo >= 0.f ? __float_as_uint(t.lo) + 1u : 0u;
            const uint32_t far = __reduce_max_sync(0xFFFFFFFFu, key);
            const unsigned at_far = __ballot_sync(0xFFFFFFFFu, key == far);
            const int wl = __ffs(at_far) - 1;
            const float bar = __uint_as_float(far - 1u);
            const bool rival = lane < kWarps && (lane == wl ? t.hi_others : fmaxf(t.hi, t.hi_others)) >= bar;
            if (!__any_sync(0xFFFFFFFFu, rival)) {
                rep = __shfl_sync(0xFFFFFFFFu, t.row, wl);
            } else {
                // the rows that may be the farthest, by their fp64 distance to the nearest representative (kept: rows that
                // tie are asked again at the next choice)
                maybe = 0u;
#pragma unroll
                for (int k = 0; k < kRpt; ++k)
                    if ((((live & ~is_rep) >> k) & 1u) && !(hi[k] < bar)) maybe |= 1u << k;
                const int n_open = __syncthreads_count((maybe & open_owner) != 0u);
                spent += kChoiceCost + n_open * ((u + 31) / 32);
                if (spent > budget) { select_large_exact<kWarps, kRpt, kHalf>(sm, nC, r); return; }
                ValIdx x = {-2.0, INT_MAX};
#pragma unroll
                for (int k = 0; k < kRpt; ++k) {
                    double &near = sm.near[LARGE_ROW(k)];
                    bool asked = ((maybe & ~open_owner & ~known) >> k) & 1u;
                    if (asked) near = exact_dist<kHalf>(sm.rows + LARGE_ROW(k) * kPitch, sm.rows + sm.rep_of[owner[k]] * kPitch, kWords);
                    for (unsigned left = __ballot_sync(0xFFFFFFFFu, ((maybe & open_owner) >> k) & 1u); left; left &= left - 1) {
                        const int l = __ffs(left) - 1;
                        double dist;
                        const int who = nearest_rep<kHalf>(sm, warp * 32 * kRpt + 32 * k + l, u, dist);
                        if (lane == l) { near = dist; owner[k] = who; asked = true; }
                    }
                    if (asked) {                              // certain from here on, and within a float's rounding
                        lo[k] = __double2float_rd(near);
                        mind[k] = hi[k] = __double2float_ru(near);
                    }
                    if ((maybe >> k) & 1u) x = pick<false>(x, {near, LARGE_ROW(k)});
                }
                open_owner &= ~maybe;
                known |= maybe;
                x = block_arg<false>(x, sm.arg);
                rep = min(x.i, nC - 1);
            }
#pragma unroll
            for (int k = 0; k < kRpt; ++k)
                if (LARGE_ROW(k) == rep) is_rep |= 1u << k;
            const unsigned at = __ballot_sync(0xFFFFFFFFu, cand == rep);
            if (!at) break;
            col = __ffs(at) - 1;
        }
        if (done) break;
    }
    // rows whose two nearest representatives the bound leaves open: lanes take the representatives
    __syncthreads();
    const unsigned ask = live & open_owner & ~is_rep;
    if (__syncthreads_count(ask != 0u) * ((r + 31) / 32) > r * kRpt * kWarps) { select_large_exact<kWarps, kRpt, kHalf>(sm, nC, r); return; }
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        for (unsigned left = __ballot_sync(0xFFFFFFFFu, (ask >> k) & 1u); left; left &= left - 1) {
            const int l = __ffs(left) - 1;
            double dist;
            const int who = nearest_rep<kHalf>(sm, warp * 32 * kRpt + 32 * k + l, r, dist);
            if (lane == l) owner[k] = who;
        }
        sm.owner[LARGE_ROW(k)] = (uint16_t)owner[k];
    }
    __syncthreads();
}

template <int kWarps, int kRpt, bool kHalf>
__device__ __forceinline__ void large_parent(const ParentRows &t, LargeSmem<kWarps, kRpt> &sm)
{
    using Smem = LargeSmem<kWarps, kRpt>;
    constexpr int kT = 32 * kWarps, kGroups = kWarps * kRpt;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, q = lane & 15;
    const uint4 *k = reinterpret_cast<const uint4 *>(t.k_prompt) + t.plane * 16;
    const uint4 *v = reinterpret_cast<const uint4 *>(t.v_prompt) + t.plane * 16;
    for (int i = tid; i < t.nC; i += kT) sm.token[i] = t.members ? t.members[i] : t.s0 + i;
    if (t.members) __syncthreads();
    for (int e = tid; e < t.nC * 16; e += kT) {
        const int i = e >> 4;
        copy16_async(shared_addr(sm.rows + i * kPitch + (e & 15) * 4), k + (size_t)(t.members ? sm.token[i] : t.s0 + i) * 16 + (e & 15));
    }
    if (!t.members && tid == 0)                              // V is read when the owners are known: into L2 meanwhile
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(v + (size_t)t.s0 * 16), "r"((uint32_t)t.nC * 256u) : "memory");
    copy_async_wait();
    __syncthreads();
    select_large<kWarps, kRpt, kHalf>(sm, t.nC, t.r);

    for (int u = tid; u < t.r; u += kT) sm.owner[sm.rep_of[u]] = (uint16_t)u;   // a representative owns its own row
    for (int e = tid; e < kGroups * t.r; e += kT) sm.count[e / t.r][e % t.r] = 0;
    __syncthreads();
    // packed order: teams in selection order, members by index. Rank inside a group of 32 rows, then prefixes
    // over the groups and over the teams.
    int owner[kRpt], rank[kRpt], pos[kRpt];
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        const bool live = LARGE_ROW(k) < t.nC;
        owner[k] = live ? sm.owner[LARGE_ROW(k)] : Smem::kRows + lane;          // idle lanes stay alone
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, owner[k]);
        rank[k] = __popc(peers & ((1u << lane) - 1u));
        if (live && rank[k] == 0) sm.count[warp * kRpt + k][owner[k]] = (uint16_t)__popc(peers);
    }
    __syncthreads();
    int carry = 0;
    for (int u0 = 0; u0 < t.r; u0 += kT) {
        const int u = u0 + tid;
        int size = 0;
        if (u < t.r) {
#pragma unroll
            for (int w = 0; w < kGroups; ++w) {
                const int n = sm.count[w][u];
                sm.count[w][u] = (uint16_t)size;
                size += n;
            }
        }
        int total;
        const int start = carry + block_exclusive_scan(size, sm.scan, total);
        if (u < t.r) {
            sm.team_start[u] = start;
            t.csr[1 + u] = t.s0 + start + size;
        }
        carry += total;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {
        pos[k] = 0;
        if (LARGE_ROW(k) < t.nC) {
            pos[k] = sm.team_start[owner[k]] + sm.count[warp * kRpt + k][owner[k]] + rank[k];
            t.row_token[t.plane + t.s0 + pos[k]] = sm.token[LARGE_ROW(k)];
        }
    }
    uint4 *kdst = reinterpret_cast<uint4 *>(t.k_packed) + (t.plane + t.s0) * 16;
    uint4 *vdst = reinterpret_cast<uint4 *>(t.v_packed) + (t.plane + t.s0) * 16;
#pragma unroll
    for (int k = 0; k < kRpt; ++k) {                         // 32 rows at a time, a row per half warp
        uint4 vr[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int i = warp * 32 * kRpt + 32 * k + 2 * m + (lane >> 4);
            vr[m] = i < t.nC ? __ldg(v + (size_t)sm.token[i] * 16 + q) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int l = 2 * m + (lane >> 4), i = warp * 32 * kRpt + 32 * k + l;
            const int d = __shfl_sync(0xFFFFFFFFu, pos[k], l);
            if (i < t.nC) {
                kdst[(size_t)d * 16 + q] = *reinterpret_cast<const uint4 *>(sm.rows + i * kPitch + q * 4);
                vdst[(size_t)d * 16 + q] = vr[m];
            }
        }
    }
    uint32_t m = 0u;
    uint4 *rdst = reinterpret_cast<uint4 *>(t.rep_keys) + t.rep0 * 16;
    for (int e = tid; e < t.r * 16; e += kT) {
        const uint4 w = *reinterpret_cast<const uint4 *>(sm.rows + sm.rep_of[e >> 4] * kPitch + (e & 15) * 4);
        rdst[e] = w;
        m = max(m, max(max(magnitude2(w.x), magnitude2(w.y)), max(magnitude2(w.z), magnitude2(w.w))));
    }
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0 && m != 0u) raise_abs_max<kHalf>(t.abs_max, m);
}

}  // namespace
}  // namespace santapp
