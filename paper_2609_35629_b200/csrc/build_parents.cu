// Team records from an arbitrary parent partition (the partition Algorithm 3 returns: parents of
// any size, in centre order, empty ones omitted), and the nearest-centre assignment that closes
// Algorithm 3. Preparation path, run once after prefill. As in the contiguous builder, the teams are those of fp64
// distances summed over dimensions in increasing order with separately rounded multiply and add.
//
// Steps: rank every token among the earlier tokens of its label (per chunk of the sequence, side by side) and count
// the labels of each chunk; scan the counts into member-list offsets, number the teams (a parent of c tokens
// yields min(R, c)) and list the parents by size; write the member lists; then one kernel per size class does
// Algorithm 2 and the packed copy of its parents (parent_teams.cuh; a parent's rows are one range of the packed
// order). 4 x 32K keys in 2048 k-means parents: 1250 us with one block per pair scattering tokens in order, by
// label and again by team.
#include <limits.h>

#include <algorithm>

#include "build_util.cuh"
#include "common.cuh"
#include "nearest.cuh"
#include "parent_teams.cuh"

namespace santapp {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int clamp_label(int v, int n) { return min(max(v, 0), n - 1); }

// ---- Algorithm 3, assignment step: b_i = argmin_u |k_i - mu_u|^2, ties to the smaller u ----
// A block takes 128 tokens and scans all centres (nearest.cuh), which it rounds to 16 bits as it brings them into shared
// memory (half a row per thread). Only tokens whose bounds leave more than one centre see fp64. 4 x 32768 tokens,
// 2048 centres: 6.7 ms with every distance in fp64.
// Tokens of a block up to which they go through all centres one by one: at 512 centres eight of them, a warp each, take about 60 us,
// and a block that takes all of its tokens together 200 to 400.
constexpr int kAssignFewOpen = 24;
template <bool kHalf>
__global__ void __launch_bounds__(kNearThreads, 2)
assign_parents_kernel(AssignParams p)
{
    extern __shared__ __align__(1024) unsigned char near_smem[];
    NearSmem &sm = *reinterpret_cast<NearSmem *>(near_smem);
    step_wait();
    __shared__ int n_open;                                  // tokens that go through all centres
    const int b = blockIdx.y, j = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = p.seq_row_off[b];
    const int N = (int)(p.seq_row_off[b + 1] - row0), i0 = blockIdx.x * kNearPoints;
    if (i0 >= N) return;
    if (tid == 0) n_open = 0;
    const int64_t c0off = p.seq_centre_off[b];
    const int k = (int)(p.seq_centre_off[b + 1] - c0off);
    const uint16_t *keys = p.k_prompt + ((size_t)j * p.rows_total + row0) * kHeadDim;
    const float *cen = p.centres + ((size_t)j * p.centres_total + c0off) * kHeadDim;
    uint32_t uses[2] = {0u, 0u};
    near_open_block(sm);
    near_scan<kHalf>(sm, [&](int i) { return keys + (size_t)min(i0 + i, N - 1) * kHeadDim; }, 0, k, uses,
                     [&](int stage, int slot, int base, int n) {
        // eight lanes share a row: lane part takes pieces part and part + 8, a 32-byte run of the centre each
        const int part = tid & 7;
#pragma unroll 2
        for (int r0 = 0; r0 < kNearTile; r0 += kNearThreads / 8) {
            const int row = r0 + (tid >> 3);
            float nc = 0.f, m = 0.f;
            uint4 out[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
            if (row < n) {
                const float *src = cen + (size_t)(base + row) * kHeadDim;
                const bool wide = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float *from = src + 8 * (part + 8 * c);
                    float v[8];
                    if (wide) {
                        const float4 v0 = __ldg(reinterpret_cast<const float4 *>(from)), v1 = __ldg(reinterpret_cast<const float4 *>(from + 4));
                        v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w; v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = __ldg(from + e);
                    }
                    uint32_t hi[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        hi[e] = pack_elems<kHalf>(v[2 * e], v[2 * e + 1]);
                        const float r0v = v[2 * e] - elem_lo<kHalf>(hi[e]), r1v = v[2 * e + 1] - elem_hi<kHalf>(hi[e]);
                        nc = fmaf(v[2 * e], v[2 * e], fmaf(v[2 * e + 1], v[2 * e + 1], nc));
                        m = fmaf(r0v, r0v, fmaf(r1v, r1v, m));
                    }
                    out[c] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                }
            }
#pragma unroll
            for (int o = 1; o <= 4; o <<= 1) {
                nc += __shfl_xor_sync(0xFFFFFFFFu, nc, o);
                m += __shfl_xor_sync(0xFFFFFFFFu, m, o);
            }
            const float bias = row < n ? centre_bias<kHalf>(nc) : kNearFar;
            const bool fits = row < n && bias > -kNearFar;  // else: no part in the products
#pragma unroll
            for (int c = 0; c < 2; ++c)
                *reinterpret_cast<uint4 *>(sm.centres[stage] + near_byte(row, part + 8 * c)) = fits ? out[c] : make_uint4(0u, 0u, 0u, 0u);
            if (part == 0) sm.bias[slot][row] = make_float2(bias, fits ? 1.00001f * sqrtf(m) : 0.f);
        }
    });
    const int point = tid % kNearPoints, i = i0 + point;
    const NearTop top = sm.top[point];
    const uint4 *x = reinterpret_cast<const uint4 *>(keys + (size_t)min(i, N - 1) * kHeadDim);
    int32_t *labels = p.parent_of + (size_t)j * p.rows_total + row0;
    const bool open = i < N && near_open(top, sm.nx[point]);
    if (tid < kNearPoints && open) sm.idx[atomicAdd(&n_open, 1)] = i;
    if (tid < kNearPoints && i < N && !open) {
        int arg = top.i1;
        if (!(top.t2 > top.upper)) {
            double best = near_exact<kHalf>(x, cen + (size_t)arg * kHeadDim);
            const double d2 = near_exact<kHalf>(x, cen + (size_t)top.i2 * kHeadDim);
            if (d2 < best || (d2 == best && top.i2 < arg)) { best = d2; arg = top.i2; }
            if (!(top.t3 > top.upper)) {
                const double d3 = near_exact<kHalf>(x, cen + (size_t)top.i3 * kHeadDim);
                if (d3 < best || (d3 == best && top.i3 < arg)) { best = d3; arg = top.i3; }
            }
        }
        labels[i] = arg;
    }
    __syncthreads();
    double d;
    if (n_open > kAssignFewOpen) {
        const int arg = near_scan_tiles<kHalf, kNearThreads, 2>(x, open, cen, k, reinterpret_cast<double (*)[kHeadDim]>(sm.centres[0]), d);
        if (tid < kNearPoints && open) labels[i] = arg;
    } else {
        for (int e = warp; e < n_open; e += kNearThreads / 32) {
            const int arg = near_scan_exact<kHalf>(reinterpret_cast<const uint4 *>(keys + (size_t)sm.idx[e] * kHeadDim), cen, k,
                                                   reinterpret_cast<double *>(sm.points) + warp * kHeadDim, d);
            if (lane == 0) labels[sm.idx[e]] = arg;
        }
    }
    near_close_block(sm);
}

// At most eight centres: one pass of fp64 distances, two tokens per thread. Bound by fp64 additions, like the scan above
// where centres lie close together, but without its set-up: 4 x 100000 tokens and two or eight centres 107 us, the scan
// 130, or 180 and 250 when the centres are means of random tokens.
constexpr int kFewCentres = 8, kFewThreads = 128, kFewPoints = 2;
template <bool kHalf>
__global__ void __launch_bounds__(kFewThreads)
assign_few_kernel(AssignParams p)
{
    __shared__ __align__(16) double c[kFewCentres][kHeadDim];
    step_wait();
    const int b = blockIdx.y, j = blockIdx.z, tid = threadIdx.x;
    const int64_t row0 = p.seq_row_off[b], c0off = p.seq_centre_off[b];
    const int N = (int)(p.seq_row_off[b + 1] - row0), k = (int)(p.seq_centre_off[b + 1] - c0off), i0 = blockIdx.x * kFewPoints * kFewThreads;
    if (i0 >= N) return;
    const float *cen = p.centres + ((size_t)j * p.centres_total + c0off) * kHeadDim;
    for (int e = tid; e < kFewCentres * kHeadDim; e += kFewThreads)
        c[e / kHeadDim][e % kHeadDim] = (double)__ldg(cen + (size_t)min(e / kHeadDim, k - 1) * kHeadDim + e % kHeadDim);
    const size_t plane = (size_t)j * p.rows_total + row0;
    const uint4 *row[kFewPoints];
#pragma unroll
    for (int u = 0; u < kFewPoints; ++u)
        row[u] = reinterpret_cast<const uint4 *>(p.k_prompt + (plane + min(i0 + u * kFewThreads + tid, N - 1)) * kHeadDim);
    __syncthreads();
    double d[kFewPoints][kFewCentres] = {};
    dist_points<kHalf, kFewPoints, kFewCentres, kFewCentres>(row, c, d);
#pragma unroll
    for (int u = 0; u < kFewPoints; ++u) {
        const int i = i0 + u * kFewThreads + tid;
        double best = INFINITY;
        int arg = 0;
#pragma unroll
        for (int v = 0; v < kFewCentres; ++v)
            if (v < k && d[u][v] < best) { best = d[u][v]; arg = v; }
        if (i < N) p.parent_of[plane + i] = arg;
    }
}

// ---- member lists ----
// One warp per (chunk of a sequence's tokens, sequence, KV head): the tokens 32 at a time in increasing index; lanes with
// the same label form a group whose lowest lane moves the label's count, and each lane takes its rank in the
// group on top of the count before. The chunk's counts go to label_hist. They live in shared memory when they
// fit (smem_labels of them), else in label_hist itself; a step's labels are requested one step ahead.
constexpr int kHistSmemLabels = 50 * 1024;                  // 200 KB
constexpr int kRankThreads = 128;                           // all of them clear and write the counts, the first warp ranks
__global__ void __launch_bounds__(kRankThreads)
rank_labels_kernel(ParentBuildParams p, int smem_labels)
{
    extern __shared__ int32_t count_s[];
    step_wait();
    const int chunk = blockIdx.x, b = blockIdx.y, j = blockIdx.z, tid = threadIdx.x, lane = tid & 31;
    const int64_t row0 = p.bv.seq_row_off[b];
    const int N = (int)(p.bv.seq_row_off[b + 1] - row0);
    const int64_t l0 = p.seq_label_off[b];
    const int n_labels = (int)(p.seq_label_off[b + 1] - l0);
    const int per = ((N + p.chunks - 1) / p.chunks + 31) / 32 * 32, lo = min(chunk * per, N), hi = min(lo + per, N);
    const size_t plane = (size_t)j * p.bv.rows_total + row0;
    int32_t *hist = p.label_hist + ((size_t)j * p.chunks + chunk) * p.labels_total + l0;
    const bool in_smem = n_labels <= smem_labels;
    int32_t *count = in_smem ? count_s : hist;
    for (int u = tid; u < n_labels; u += kRankThreads) count[u] = 0;
    __syncthreads();
    if (tid < 32) {
        const int32_t *lab = p.parent_of + plane;
        int next = lo + lane < hi ? lab[lo + lane] : 0;
        for (int i0 = lo; i0 < hi; i0 += 32) {
            const int i = i0 + lane, mine = next;
            const bool valid = i < hi;
            if (i + 32 < hi) next = lab[i + 32];
            const int u = valid ? clamp_label(mine, n_labels) : -1 - lane;     // idle lanes stay alone
            const unsigned group = __match_any_sync(0xFFFFFFFFu, u);
            const int leader = __ffs(group) - 1;
            int base = 0;
            if (valid && lane == leader) base = atomicAdd(count + u, __popc(group));
            base = __shfl_sync(0xFFFFFFFFu, base, leader);  // (also completes a step's updates before the next)
            if (valid) p.rank[plane + i] = base + __popc(group & ((1u << lane) - 1u));
        }
    }
    __syncthreads();
    if (in_smem)
        for (int u = tid; u < n_labels; u += kRankThreads) hist[u] = count_s[u];
}

// One block per (sequence, KV head): counts of the chunks -> where each chunk's tokens of a label go in the member
// list, member-list offsets, team numbering, team count, the row offsets of the slots behind the last team (empty
// teams), and the parents by size class.
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads)
scan_parents_kernel(ParentBuildParams p)
{
    __shared__ int scratch[33];
    step_wait();
    const int b = blockIdx.x, j = blockIdx.y, tid = threadIdx.x;
    const int64_t l0 = p.seq_label_off[b];
    const int n_labels = (int)(p.seq_label_off[b + 1] - l0);
    int32_t *tbase = p.parent_team_base + (size_t)j * p.labels_total + l0;
    int32_t *pstart = p.parent_start + (size_t)j * (p.labels_total + p.bv.n_seqs) + l0 + b;
    int rows_carry = 0, teams_carry = 0;
    for (int base = 0; base < n_labels; base += kScanThreads) {
        const int u = base + tid;
        int32_t *hist = p.label_hist + (size_t)j * p.chunks * p.labels_total + l0 + u;
        int cnt = 0;
        if (u < n_labels)
            for (int c0 = 0; c0 < p.chunks; c0 += 8) {
                int h[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) h[c] = c0 + c < p.chunks ? hist[(size_t)(c0 + c) * p.labels_total] : 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (c0 + c < p.chunks) hist[(size_t)(c0 + c) * p.labels_total] = cnt;
                    cnt += h[c];
                }
            }
        int rows_total, teams_total;
        const int rows_excl = block_exclusive_scan(cnt, scratch, rows_total);
        const int teams_excl = block_exclusive_scan(min(cnt, p.reps), scratch, teams_total);
        if (u < n_labels) {
            pstart[u] = rows_carry + rows_excl;
            tbase[u] = teams_carry + teams_excl;
            const int kind = p.mean_keys ? -1 : (cnt <= 32 ? -1 : (cnt <= 128 ? 0 : (cnt <= 512 ? 1 : 2)));
            if (kind >= 0) p.list[kind][atomicAdd(p.list_count + kind, 1)] = make_int2(b * p.bv.n_kv + j, u);
        }
        rows_carry += rows_total;
        teams_carry += teams_total;
    }
    const int64_t team0 = p.bv.seq_team_off[b];
    const int slots = (int)(p.bv.seq_team_off[b + 1] - team0);
    const int N = (int)(p.bv.seq_row_off[b + 1] - p.bv.seq_row_off[b]);
    int32_t *csr = p.team_row_start + (size_t)j * (p.bv.teams_total + p.bv.n_seqs) + team0 + b;
    for (int g = teams_carry + tid; g < slots; g += kScanThreads) csr[1 + g] = N;
    if (tid == 0) {
        pstart[n_labels] = rows_carry;
        p.team_count[(size_t)j * p.bv.n_seqs + b] = teams_carry;
        csr[0] = 0;
    }
}

__global__ void __launch_bounds__(kThreads)
members_kernel(ParentBuildParams p)
{
    step_wait();
    const int b = blockIdx.y, j = blockIdx.z;
    const int64_t row0 = p.bv.seq_row_off[b];
    const int N = (int)(p.bv.seq_row_off[b + 1] - row0), i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= N) return;
    const int64_t l0 = p.seq_label_off[b];
    const int n_labels = (int)(p.seq_label_off[b + 1] - l0);
    const int per = ((N + p.chunks - 1) / p.chunks + 31) / 32 * 32;
    const size_t plane = (size_t)j * p.bv.rows_total + row0;
    const int u = clamp_label(p.parent_of[plane + i], n_labels);
    const int at = p.parent_start[(size_t)j * (p.labels_total + p.bv.n_seqs) + l0 + b + u]
                   + p.label_hist[((size_t)j * p.chunks + i / per) * p.labels_total + l0 + u] + p.rank[plane + i];
    p.members[plane + at] = i;
}

// The parent of label u of (sequence b, KV head j).
__device__ __forceinline__ void listed_parent(const ParentBuildParams &p, int u, int b, int j, ParentRows &t)
{
    const int64_t l0 = p.seq_label_off[b], row0 = p.bv.seq_row_off[b], team0 = p.bv.seq_team_off[b];
    const int32_t *pstart = p.parent_start + (size_t)j * (p.labels_total + p.bv.n_seqs) + l0 + b;
    const int tb = p.parent_team_base[(size_t)j * p.labels_total + l0 + u];
    t.k_prompt = p.k_prompt;
    t.v_prompt = p.v_prompt;
    t.k_packed = p.k_packed;
    t.v_packed = p.v_packed;
    t.rep_keys = p.rep_keys;
    t.row_token = p.row_token;
    t.plane = (size_t)j * p.bv.rows_total + row0;
    t.s0 = pstart[u];
    t.nC = pstart[u + 1] - t.s0;
    t.r = min(p.reps, t.nC);
    t.members = p.members + t.plane + t.s0;
    t.csr = p.team_row_start + (size_t)j * (p.bv.teams_total + p.bv.n_seqs) + team0 + b + tb;
    t.rep0 = (size_t)j * p.bv.teams_total + team0 + tb;
    t.abs_max = p.rep_abs_max + (size_t)j * p.bv.n_seqs + b;
}

// Parents of at most 32 rows, a warp per label.
constexpr int kSmallParentWarps = 2;
template <bool kHalf>
__global__ void __launch_bounds__(kSmallParentWarps * 32)
small_parents_kernel(ParentBuildParams p)
{
    __shared__ union { SmallSmem<16> s16; SmallSmem<32> s32; } sm[kSmallParentWarps];
    step_wait();
    const int warp = threadIdx.x >> 5, u = blockIdx.x * kSmallParentWarps + warp, b = blockIdx.y, j = blockIdx.z;
    if (u >= (int)(p.seq_label_off[b + 1] - p.seq_label_off[b])) return;
    ParentRows t;
    listed_parent(p, u, b, j, t);
    if (t.nC == 0 || t.nC > 32) return;                     // empty parents are omitted
    if (t.nC <= 16) small_parent<16, kHalf>(t, sm[warp].s16);
    else            small_parent<32, kHalf>(t, sm[warp].s32);
}

// Parents of 33 to 128 and of 129 to 512 rows: blocks walk the lists.
template <int kWarps, int kRpt, bool kHalf>
__global__ void __launch_bounds__(32 * kWarps, large_blocks(kWarps, kRpt))
large_parents_kernel(ParentBuildParams p, int kind)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    step_wait();
    const int n = p.list_count[kind];
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int2 e = p.list[kind][i];
        ParentRows t;
        listed_parent(p, e.y, e.x / p.bv.n_kv, e.x % p.bv.n_kv, t);
        large_parent<kWarps, kRpt, kHalf>(t, *reinterpret_cast<LargeSmem<kWarps, kRpt> *>(smem_raw));
        __syncthreads();
    }
}

// K and V of up to 32 tokens (one per lane, the first n of them) to rows of the sequence's packed order, by a warp: eight
// tokens are on their way at a time, a half warp each. (One at a time, a block took 7 ms for 50000 tokens.)
__device__ __forceinline__ void copy_rows(const ParentRows &t, int token, int row, int n)
{
    const int lane = threadIdx.x & 31, q = lane & 15;
    const uint4 *k = reinterpret_cast<const uint4 *>(t.k_prompt) + t.plane * 16 + q, *v = reinterpret_cast<const uint4 *>(t.v_prompt) + t.plane * 16 + q;
    uint4 *kd = reinterpret_cast<uint4 *>(t.k_packed) + t.plane * 16 + q, *vd = reinterpret_cast<uint4 *>(t.v_packed) + t.plane * 16 + q;
    for (int l0 = 0; l0 < n; l0 += 8) {
        uint4 kr[4], vr[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int l = l0 + 2 * m + (lane >> 4);
            const size_t at = (size_t)__shfl_sync(0xFFFFFFFFu, token, l) * 16;
            if (l < n) { kr[m] = __ldg(k + at); vr[m] = __ldg(v + at); }
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int l = l0 + 2 * m + (lane >> 4);
            const size_t at = (size_t)__shfl_sync(0xFFFFFFFFu, row, l) * 16;
            if (l < n) { kd[at] = kr[m]; vd[at] = vr[m]; }
        }
    }
    if (lane < n) t.row_token[t.plane + row] = token;
}

template <bool kHalf>
__device__ __forceinline__ double sqdist_grow_vec(const uint4 *row, const double *ref)
{
    double s = 0.0;
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
        const uint4 w4 = row[q];
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double e0 = __dsub_rn((double)elem_lo<kHalf>(w[t]), ref[8 * q + 2 * t]);
            const double e1 = __dsub_rn((double)elem_hi<kHalf>(w[t]), ref[8 * q + 2 * t + 1]);
            s = __dadd_rn(s, __dmul_rn(e0, e0));
            s = __dadd_rn(s, __dmul_rn(e1, e1));
        }
    }
    return s;
}

template <bool kHalf>
__device__ __forceinline__ double sqdist_grow_row(const uint4 *row, const uint32_t *ref)
{
    double s = 0.0;
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
        const uint4 w4 = row[q];
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t r = ref[4 * q + t];
            const double e0 = __dsub_rn((double)elem_lo<kHalf>(w[t]), (double)elem_lo<kHalf>(r));
            const double e1 = __dsub_rn((double)elem_hi<kHalf>(w[t]), (double)elem_hi<kHalf>(r));
            s = __dadd_rn(s, __dmul_rn(e0, e0));
            s = __dadd_rn(s, __dmul_rn(e1, e1));
        }
    }
    return s;
}

// Parents of more than 512 rows (and, for the centroid-guided baseline, all parents): rows are read through the member
// list, the per-member state lives in global memory, every distance is taken in fp64. Blocks walk the list
// of such parents (mean keys: one block per label).
constexpr int kHugeBlocks = 2;          // per SM; with three or four the inner loops lack registers (8 % slower where each has a parent)
template <bool kHalf>
__global__ void __launch_bounds__(kThreads, kHugeBlocks)
huge_parents_kernel(ParentBuildParams p)
{
    __shared__ int scan_s[33], start_s[kMaxParent];
    __shared__ double mu[kHeadDim];
    __shared__ uint32_t ref[64];
    __shared__ ValIdx scratch[33];
    __shared__ int count[kMaxParent];
    __shared__ int rep_pos[kMaxParent];
    step_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_list = p.mean_keys ? 0 : p.list_count[2];
  for (int li = blockIdx.x; p.mean_keys ? li == (int)blockIdx.x : li < n_list; li += gridDim.x) {
    int u_parent = blockIdx.x, b = blockIdx.y, j = blockIdx.z;
    if (!p.mean_keys) {
        const int2 e = p.list[2][li];
        u_parent = e.y;
        b = e.x / p.bv.n_kv;
        j = e.x % p.bv.n_kv;
    } else if (u_parent >= (int)(p.seq_label_off[b + 1] - p.seq_label_off[b])) {
        return;
    }
    ParentRows t;
    listed_parent(p, u_parent, b, j, t);
    const int s0 = t.s0, nC = t.nC, r = t.r;
    if (nC == 0) return;                                   // (mean keys) empty parents are omitted
    const size_t plane = t.plane;
    const int32_t *mem = t.members;
    __syncthreads();
    double *mind = p.mind + plane + s0;
    int32_t *owner = p.owner + plane + s0;
    unsigned char *is_rep = p.is_rep + plane + s0;
    const uint4 *kbase = reinterpret_cast<const uint4 *>(p.k_prompt + plane * kHeadDim);   // 16 per row

    for (int i = tid; i < nC; i += kThreads) { is_rep[i] = 0; mind[i] = INFINITY; owner[i] = 0; }
    for (int u = tid; u < r; u += kThreads) count[u] = 0;

    // parent mean: rows added in token order, then one division
    if (tid < kHeadDim) {
        const uint16_t *col = p.k_prompt + plane * kHeadDim + tid;
        double s = 0.0;
        for (int i = 0; i < nC; ++i) s = __dadd_rn(s, elem_to_double<kHalf>(col[(size_t)mem[i] * kHeadDim]));
        mu[tid] = __ddiv_rn(s, (double)nC);
    }
    __syncthreads();

    if (p.mean_keys) {
        // centroid-guided baseline: the parent is one group, routed by its mean stored as a 16-bit
        // element (fp64 -> fp32 to nearest, fp32 -> bf16 or fp16 to nearest even)
        if (tid == 0) t.csr[1] = s0 + nC;
        if (tid < kHeadDim) p.rep_keys[t.rep0 * kHeadDim + tid] = double_to_elem<kHalf>(mu[tid]);
        for (int i = 32 * warp; i < nC; i += kThreads) copy_rows(t, mem[min(i + lane, nC - 1)], s0 + i + lane, min(32, nC - i));
        return;
    }

    // first representative: the actual key nearest the mean
    {
        ValIdx best = {INFINITY, INT_MAX};
        for (int i = tid; i < nC; i += kThreads) {
            const double d = sqdist_grow_vec<kHalf>(kbase + (size_t)mem[i] * 16, mu);
            best = pick<true>(best, {d == d ? d : INFINITY, i});       // (not a number counts as infinitely far)
        }
        best = block_arg<true>(best, scratch);
        if (tid == 0) { rep_pos[0] = best.i; is_rep[best.i] = 1; }
    }
    __syncthreads();

    // farthest-first representatives; the running (nearest distance, owner) pair is the
    // nearest-representative assignment with ties going to the earlier-selected one
    for (int u = 0; u < r; ++u) {
        if (tid < 64) ref[tid] = reinterpret_cast<const uint32_t *>(kbase + (size_t)mem[rep_pos[u]] * 16)[tid];
        __syncthreads();
        ValIdx far = {-2.0, INT_MAX};
        for (int i = tid; i < nC; i += kThreads) {
            const double dist = sqdist_grow_row<kHalf>(kbase + (size_t)mem[i] * 16, ref);
            double m = mind[i];
            if (dist < m) { m = dist; mind[i] = dist; owner[i] = u; }
            ValIdx c = {is_rep[i] ? -1.0 : m, i};
            far = pick<false>(far, c);
        }
        if (u + 1 < r) {
            far = block_arg<false>(far, scratch);
            if (tid == 0) { rep_pos[u + 1] = far.i; is_rep[far.i] = 1; }
        }
        __syncthreads();
    }
    // representative self-ownership
    for (int u = tid; u < r; u += kThreads) owner[rep_pos[u]] = u;
    __syncthreads();
    for (int i = tid; i < nC; i += kThreads) atomicAdd(&count[owner[i]], 1);
    __syncthreads();

    // team sizes -> row offsets; then the rows in member order, a warp's 32 at a time, each at its team's cursor
    int carry = 0;
    for (int u0 = 0; u0 < r; u0 += kThreads) {
        const int u = u0 + tid, n = u < r ? count[u] : 0;
        int total;
        const int start = carry + block_exclusive_scan(n, scan_s, total);
        if (u < r) {
            start_s[u] = start;
            t.csr[1 + u] = s0 + start + n;
        }
        carry += total;
    }
    __syncthreads();
    for (int i0 = 0; i0 < nC; i0 += kThreads) {
        const int i = i0 + tid;
        const int own = i < nC ? owner[i] : kMaxParent + lane;    // idle lanes stay alone
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, own);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        int pos = 0;
        for (int w = 0; w < kThreads / 32; ++w) {
            if (w == warp) {
                if (i < nC) pos = start_s[own] + rank;
                __syncwarp();
                if (i < nC && rank == 0) start_s[own] += __popc(peers);
            }
            __syncthreads();
        }
        copy_rows(t, mem[min(i, nC - 1)], s0 + pos, min(32, nC - (i0 + warp * 32)));
    }
    uint32_t m = 0u;
    uint32_t *rep_dst = reinterpret_cast<uint32_t *>(p.rep_keys) + t.rep0 * 64;
    for (int e = tid; e < r * 64; e += kThreads) {
        const uint32_t w = reinterpret_cast<const uint32_t *>(kbase + (size_t)mem[rep_pos[e >> 6]] * 16)[e & 63];
        rep_dst[e] = w;
        m = max(m, magnitude2(w));
    }
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0) raise_abs_max<kHalf>(t.abs_max, m);
  }
}

}  // namespace

template <bool kHalf>
static cudaError_t launch_assign(const AssignParams &p, cudaStream_t s)
{
    if (p.max_centres_per_seq <= kFewCentres)
        return launch_step(assign_few_kernel<kHalf>, dim3((p.max_rows_per_seq + kFewPoints * kFewThreads - 1) / (kFewPoints * kFewThreads), p.n_seqs, p.n_kv),
                           dim3(kFewThreads), 0, s, p);
    static std::atomic<unsigned long long> done;
    const cudaError_t err = ensure_dynamic_smem((const void *)assign_parents_kernel<kHalf>, (int)sizeof(NearSmem), done);
    if (err != cudaSuccess) return err;
    return launch_step(assign_parents_kernel<kHalf>, dim3((p.max_rows_per_seq + kNearPoints - 1) / kNearPoints, p.n_seqs, p.n_kv),
                       dim3(kNearThreads), sizeof(NearSmem), s, p);
}
cudaError_t launch_assign_parents(const AssignParams &p, cudaStream_t s)
{
    return p.elem ? launch_assign<true>(p, s) : launch_assign<false>(p, s);
}

template <bool kHalf>
static cudaError_t launch_parents(const ParentBuildParams &p, cudaStream_t s)
{
    const int B = p.bv.n_seqs, H = p.bv.n_kv, sms = attend_grid_size();
    cudaError_t err;
    if (p.mean_keys) return launch_step(huge_parents_kernel<kHalf>, dim3(p.max_labels_per_seq, B, H), dim3(kThreads), 0, s, p);
    // the few large parents first: theirs are the longest blocks. As many as are resident: a parent is a chain of reads
    // that one block cannot keep an SM busy with (8 sequences of 32K tokens in 40 parents per KV head: 7.4 ms at one
    // per SM, 3.6 at two, 4.1 with a block per parent)
    if ((err = launch_step(huge_parents_kernel<kHalf>, dim3(kHugeBlocks * sms), dim3(kThreads), 0, s, p)) != cudaSuccess) return err;
    static std::atomic<unsigned long long> large_done, mid_done;
    using Large = LargeSmem<8, 2>;
    using Mid = LargeSmem<4, 1>;
    if ((err = ensure_dynamic_smem((const void *)large_parents_kernel<8, 2, kHalf>, (int)sizeof(Large), large_done)) != cudaSuccess) return err;
    if ((err = ensure_dynamic_smem((const void *)large_parents_kernel<4, 1, kHalf>, (int)sizeof(Mid), mid_done)) != cudaSuccess) return err;
    if ((err = launch_step(large_parents_kernel<8, 2, kHalf>, dim3(sms), dim3(256), sizeof(Large), s, p, 1)) != cudaSuccess) return err;
    if ((err = launch_step(large_parents_kernel<4, 1, kHalf>, dim3(large_blocks(4, 1) * sms), dim3(128), sizeof(Mid), s, p, 0)) != cudaSuccess) return err;
    return launch_step(small_parents_kernel<kHalf>, dim3((p.max_labels_per_seq + kSmallParentWarps - 1) / kSmallParentWarps, B, H),
                       dim3(kSmallParentWarps * 32), 0, s, p);
}

cudaError_t launch_build_teams_parents(const ParentBuildParams &p, cudaStream_t s)
{
    const int B = p.bv.n_seqs, H = p.bv.n_kv;
    cudaError_t err = cudaMemsetAsync(p.list_count, 0, sizeof(int32_t) * 3, s);
    if (err != cudaSuccess) return err;
    // representative keys of the empty slots are zero
    err = cudaMemsetAsync(p.rep_keys, 0, sizeof(uint16_t) * (size_t)H * p.bv.teams_total * kHeadDim, s);
    if (err != cudaSuccess) return err;
    static std::atomic<unsigned long long> rank_done;
    const int smem_labels = std::min(p.max_labels_per_seq, kHistSmemLabels);
    if ((err = ensure_dynamic_smem((const void *)rank_labels_kernel, (int)sizeof(int32_t) * kHistSmemLabels, rank_done)) != cudaSuccess) return err;
    if ((err = launch_step(rank_labels_kernel, dim3(p.chunks, B, H), dim3(kRankThreads), sizeof(int32_t) * (size_t)smem_labels, s, p, smem_labels)) != cudaSuccess)
        return err;
    if ((err = launch_step(scan_parents_kernel, dim3(B, H), dim3(kScanThreads), 0, s, p)) != cudaSuccess) return err;
    if ((err = launch_step(members_kernel, dim3((p.max_rows_per_seq + kThreads - 1) / kThreads, B, H), dim3(kThreads), 0, s, p)) != cudaSuccess) return err;
    return p.bv.elem ? launch_parents<true>(p, s) : launch_parents<false>(p, s);
}

}  // namespace santapp
