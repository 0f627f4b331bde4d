// santapp_kmeans_fit: the fit of Algorithm 3 (global minibatch k-means parents), one independent
// problem per (sequence, KV head). Preparation path, run once after prefill.
//
// The paper names the routine and its settings and leaves the rest to its library; the reading
// taken here is written out in include/santapp.h. Every random choice is a Philox word with
// counter (slot, tag, stream, step), and every comparison is made on fp64 values obtained by the
// same operations in the same order wherever the order matters (sums over dimensions, over the
// sample, over a minibatch; separately rounded multiply and add), so a fit is a pure function
// of its arguments. Sums whose order matters run on one thread; the distance evaluations around
// them are spread over the grid.
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "nearest.cuh"

namespace santapp {

namespace {

constexpr int kThreads = 256;
constexpr int kPollEvery = 16;            // steps between two looks at the fits' stop flags
constexpr uint32_t kTagSample = 1u, kTagStart = 2u, kTagBatch = 3u, kTagMove = 4u;

struct Pair {
    int b, j, N, k, n_init, L, t_max;
    uint32_t stream;
    int64_t row0, c0;
    size_t plane;                         // first row of the pair in a [n_kv][rows_total] array
    size_t cplane;                        // first centre of the pair in a [n_kv][centres_total] array
    int id;                               // j-major pair index into the per-pair scratch arrays
};

__device__ __forceinline__ Pair pair_of(const KmeansParams &p, int b, int j)
{
    Pair q;
    q.b = b;
    q.j = j;
    q.row0 = p.seq_row_off[b];
    q.N = (int)(p.seq_row_off[b + 1] - q.row0);
    q.c0 = p.seq_centre_off[b];
    q.k = (int)(p.seq_centre_off[b + 1] - q.c0);
    q.n_init = p.seq_n_init[b];
    q.L = p.seq_trials[b];
    q.t_max = p.seq_t_max[b];
    q.stream = p.stream_base + (uint32_t)(b * p.n_kv + j);
    q.plane = (size_t)j * p.rows_total + (size_t)q.row0;
    q.cplane = (size_t)j * p.centres_total + (size_t)q.c0;
    q.id = j * p.n_seqs + b;
    return q;
}

__device__ __forceinline__ uint32_t km_word(const KmeansParams &p, uint32_t slot, uint32_t tag, uint32_t stream, uint32_t step)
{
    return philox4x32_10(make_uint4(slot, tag, stream, step), p.seed_lo, p.seed_hi).x;
}
__device__ __forceinline__ int km_index(uint32_t word, int n) { return (int)(((unsigned long long)word * (unsigned long long)n) >> 32); }

// ---- 1. initialisation sample: head of a Fisher-Yates shuffle ----
// Step i of the shuffle swaps entries i and r_i >= i of the index list, so entry i is final after step i, and holds
// what entry r_i held before it: the value that the last earlier step j with r_j = r_i put there, which is what
// entry j held before step j, and so on until no earlier step touched the entry (it still holds its own
// index). The chains are short (about one step), so every entry is found on its own: steps are looked up by
// target in a hash table in shared memory. One block per pair. (Swapping in order took 60 ns a step, 0.75 ms.)
constexpr int kSampleThreads = 1024, kSampleBuckets = 8192;
__host__ __device__ constexpr size_t sample_smem(int n_init)
{
    return sizeof(int32_t) * ((size_t)kSampleBuckets + (size_t)n_init) + sizeof(uint16_t) * (size_t)n_init;
}
__global__ void __launch_bounds__(kSampleThreads)
km_sample_kernel(KmeansParams p)
{
    extern __shared__ int32_t bucket_s[];                     // step + 1 of a bucket's first entry, 0: none
    step_wait();
    const Pair q = pair_of(p, blockIdx.x, blockIdx.y);
    const int tid = threadIdx.x;
    int32_t *target_s = bucket_s + kSampleBuckets;            // [n_init] r_i
    uint16_t *next_s = reinterpret_cast<uint16_t *>(target_s + q.n_init);   // [n_init] step + 1 of the next entry in the bucket
    for (int u = tid; u < kSampleBuckets; u += kSampleThreads) bucket_s[u] = 0;
    __syncthreads();
    for (int i = tid; i < q.n_init; i += kSampleThreads) {
        const int r = i + km_index(km_word(p, (uint32_t)i, kTagSample, q.stream, 0u), q.N - i);
        target_s[i] = r;
        next_s[i] = (uint16_t)atomicExch(&bucket_s[r & (kSampleBuckets - 1)], i + 1);
    }
    __syncthreads();
    for (int i = tid; i < q.n_init; i += kSampleThreads) {
        int at = target_s[i], before = i;
        while (true) {
            int last = -1;
            for (int e = bucket_s[at & (kSampleBuckets - 1)]; e > 0; e = next_s[e - 1])
                if (target_s[e - 1] == at && e - 1 < before && e - 1 > last) last = e - 1;
            if (last < 0) break;
            at = before = last;
        }
        p.perm[q.plane + i] = at;
    }
    if (tid == 0) p.pick[(size_t)q.id * p.trials_max] = km_index(km_word(p, 0u, kTagStart, q.stream, 0u), q.n_init);
}

// ---- 2. greedy k-means++ on the sample ----
constexpr int kSumBlock = 128;           // sums over the initialisation sample are taken in blocks of this many points
constexpr int kMaxSumBlocks = 224;       // an initialisation sample holds at most 28544 points (223 blocks)
constexpr int kDistPts = 1;              // points per thread
constexpr int kDistThreads = kSumBlock / kDistPts;   // a block covers one block of the sums
static_assert(kDistThreads % 64 == 0, "64 threads widen one candidate row");
constexpr int kDistTrials = 6;           // candidate points per block

// Distances of every sample point to the candidate points pick[0..n_cand): cand[l][i]; and, for c > 0,
// the sums of min(closest_i, cand[l][i]) over each block of kSumBlock consecutive sample points, added
// in order by one thread per candidate (the potential of a trial is the sum of its block sums in order).
template <bool kHalf>
__global__ void __launch_bounds__(kDistThreads)
km_candidate_dist_kernel(KmeansParams p, int c)
{
    __shared__ __align__(16) double y_s[kDistTrials][kHeadDim];
    __shared__ double term_s[kDistTrials][kSumBlock];
    const Pair q = pair_of(p, blockIdx.z / p.n_kv, blockIdx.z % p.n_kv);
    if (c >= q.k || blockIdx.x * kSumBlock >= q.n_init) return;
    const int L = c == 0 ? 1 : q.L;
    const int n_chunks = (L + kDistTrials - 1) / kDistTrials, per = (L + n_chunks - 1) / n_chunks;
    const int l0 = blockIdx.y * per, cn = min(per, L - l0);
    if (cn <= 0) return;
    const int tid = threadIdx.x;
    const int32_t *perm = p.perm + q.plane;
    const uint16_t *keys = p.k_prompt + q.plane * kHeadDim;
    __shared__ int row_s[kDistTrials];
    if (tid < cn) row_s[tid] = perm[p.pick[(size_t)q.id * p.trials_max + l0 + tid]];
    int i[kDistPts];
    const uint4 *row[kDistPts];
#pragma unroll
    for (int j = 0; j < kDistPts; ++j) {
        i[j] = blockIdx.x * kSumBlock + j * kDistThreads + tid;
        row[j] = reinterpret_cast<const uint4 *>(keys + (size_t)perm[min(i[j], q.n_init - 1)] * kHeadDim);
    }
    __syncthreads();
    {
        // the candidates' rows as doubles: a thread widens one packed word (two values) of every
        // kGroups-th row
        constexpr int kGroups = kDistThreads / 64, kMine = (kDistTrials + kGroups - 1) / kGroups;
        const int wi = tid & 63, v0 = tid >> 6;
        uint32_t yw[kMine];
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
            const int v = v0 + m * kGroups;
            yw[m] = v < cn ? reinterpret_cast<const uint32_t *>(keys + (size_t)row_s[v] * kHeadDim)[wi] : 0u;
        }
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
            const int v = v0 + m * kGroups;
            if (v < cn) {
                y_s[v][2 * wi] = (double)elem_lo<kHalf>(yw[m]);
                y_s[v][2 * wi + 1] = (double)elem_hi<kHalf>(yw[m]);
            }
        }
    }
    __syncthreads();
    double d[kDistPts][kDistTrials];
#pragma unroll
    for (int j = 0; j < kDistPts; ++j)
#pragma unroll
        for (int v = 0; v < kDistTrials; ++v) d[j][v] = 0.0;
    switch (cn) {
    case 1: dist_points<kHalf, kDistPts, 1, kDistTrials>(row, y_s, d); break;
    case 2: dist_points<kHalf, kDistPts, 2, kDistTrials>(row, y_s, d); break;
    case 3: dist_points<kHalf, kDistPts, 3, kDistTrials>(row, y_s, d); break;
    case 4: dist_points<kHalf, kDistPts, 4, kDistTrials>(row, y_s, d); break;
    case 5: dist_points<kHalf, kDistPts, 5, kDistTrials>(row, y_s, d); break;
    default: dist_points<kHalf, kDistPts, 6, kDistTrials>(row, y_s, d); break;
    }
#pragma unroll
    for (int j = 0; j < kDistPts; ++j) {
#pragma unroll
        for (int v = 0; v < kDistTrials; ++v) {
            if (v >= cn) continue;
            double term = -1.0;                             // marks a point past the end of the sample
            if (i[j] < q.n_init) {
                p.cand[((size_t)q.id * p.trials_max + l0 + v) * p.n_init_max + i[j]] = d[j][v];
                if (c > 0) {
                    const double o = p.closest[(size_t)q.id * p.n_init_max + i[j]];
                    term = d[j][v] < o ? d[j][v] : o;
                }
            }
            term_s[v][j * kDistThreads + tid] = term;
        }
    }
    if (c == 0) return;
    __syncthreads();
    if (tid < cn) {
        double w = 0.0;
#pragma unroll 8
        for (int u = 0; u < kSumBlock; ++u) {
            const double v = term_s[tid][u];
            if (v >= 0.0) w = __dadd_rn(w, v);
        }
        const int n_part = (p.n_init_max + kSumBlock - 1) / kSumBlock;
        p.part[((size_t)q.id * p.trials_max + l0 + tid) * n_part + blockIdx.x] = w;
    }
}

constexpr int kAcceptThreads = 1024;

// One block per pair: potentials of the trials (sums in blocks of kSumBlock sample points), the best
// trial becomes centre c, the nearest-centre distances are lowered, and the trial points of centre
// c + 1 are drawn. Every serial sum runs over shared memory with its loads ahead of its additions.
template <bool kHalf>
__global__ void __launch_bounds__(kAcceptThreads)
km_accept_kernel(KmeansParams p, int c)
{
    extern __shared__ double cum_s[];                       // [n_init + blocks] running sums, then [blocks] block offsets
    __shared__ int best_s;
    __shared__ double pot_s[32];
    const Pair q = pair_of(p, blockIdx.x, blockIdx.y);
    if (c >= q.k) return;
    const int tid = threadIdx.x;
    const int n_trials = c == 0 ? 1 : q.L;
    const int n_blocks = (q.n_init + kSumBlock - 1) / kSumBlock, n_part = (p.n_init_max + kSumBlock - 1) / kSumBlock;
    double *closest = p.closest + (size_t)q.id * p.n_init_max;
    const double *cand = p.cand + (size_t)q.id * p.trials_max * p.n_init_max;
    double *off_s = cum_s + p.n_init_max + kMaxSumBlocks;
    if (c > 0) {
        // the potential of a trial: its block sums (left by the distance kernel) added in order
        for (int e = tid; e < n_trials * n_blocks; e += kAcceptThreads) {
            const int l = e / n_blocks;
            cum_s[e] = p.part[((size_t)q.id * p.trials_max + l) * n_part + (e - l * n_blocks)];
        }
        __syncthreads();
        if (tid < n_trials) {
            double pot = 0.0;
#pragma unroll 8
            for (int blk = 0; blk < n_blocks; ++blk) pot = __dadd_rn(pot, cum_s[tid * n_blocks + blk]);
            pot_s[tid] = pot;
        }
    }
    __syncthreads();
    if (tid == 0) {
        int best = 0;
        for (int l = 1; l < n_trials; ++l)
            if (pot_s[l] < pot_s[best]) best = l;
        best_s = best;
    }
    __syncthreads();
    const int best = best_s;
    const double *win = cand + (size_t)best * p.n_init_max;
    if (tid < kHeadDim) {
        const int32_t *perm = p.perm + q.plane;
        const int at = p.pick[(size_t)q.id * p.trials_max + best];
        const uint16_t v = p.k_prompt[(q.plane + (size_t)perm[at]) * kHeadDim + tid];
        p.centres64[(q.cplane + (size_t)c) * kHeadDim + tid] = elem_to_double<kHalf>(v);
    }
    // The nearest-centre distances are lowered and kept in shared memory for the draw of the next
    // centre's trial points (inverse CDF over the sample in order). cum_s holds one pad word per
    // block of the sums (point i at i + i / kSumBlock), so that threads that walk different blocks do
    // not meet in one bank.
    for (int i0 = 0; i0 < q.n_init; i0 += 8 * kAcceptThreads) {
        double d[8], o[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int i = i0 + v * kAcceptThreads + tid;
            if (i < q.n_init) {
                d[v] = win[i];
                o[v] = c == 0 ? 0.0 : closest[i];
            }
        }
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int i = i0 + v * kAcceptThreads + tid;
            if (i < q.n_init) {
                const double t = (c == 0 || d[v] < o[v]) ? d[v] : o[v];
                closest[i] = t;
                cum_s[i + i / kSumBlock] = t;
            }
        }
    }
    if (c + 1 >= q.k) return;                               // the pair's last centre draws nothing
    __syncthreads();
    // running sums inside each block (a thread per block), the block offsets in order, offset + running sum
    if (tid < n_blocks) {
        const int lo = tid * kSumBlock, cnt = min(kSumBlock, q.n_init - lo);
        double *blk_s = cum_s + lo + tid;
        double w = 0.0;
        for (int u = 0; u < cnt; u += 8) {
            double t[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) t[v] = u + v < cnt ? blk_s[u + v] : 0.0;
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                if (u + v < cnt) {
                    w = __dadd_rn(w, t[v]);
                    blk_s[u + v] = w;
                }
            }
        }
        off_s[tid] = w;
    }
    __syncthreads();
    if (tid == 0) {                                         // sums of the earlier blocks, in order
        double off = 0.0;
#pragma unroll 8
        for (int blk = 0; blk < n_blocks; ++blk) {
            const double t = off_s[blk];
            off_s[blk] = off;
            off = __dadd_rn(off, t);
        }
    }
    __syncthreads();
    for (int i = tid; i < q.n_init; i += kAcceptThreads) cum_s[i + i / kSumBlock] = __dadd_rn(off_s[i / kSumBlock], cum_s[i + i / kSumBlock]);
    __syncthreads();
    if (tid < q.L) {
        const double total = cum_s[q.n_init - 1 + (q.n_init - 1) / kSumBlock];
        const uint32_t w = km_word(p, (uint32_t)tid, kTagStart, q.stream, (uint32_t)(c + 1));
        const double target = __dmul_rn(((double)w + 0.5) * (1.0 / 4294967296.0), total);
        int lo = 0, hi = q.n_init;                          // first i in [lo, hi) with cum_s[i] > target
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (cum_s[mid + mid / kSumBlock] > target) hi = mid; else lo = mid + 1;
        }
        p.pick[(size_t)q.id * p.trials_max + tid] = lo < q.n_init ? lo : q.n_init - 1;
    }
}

// ---- 3. minibatch steps ----
// A step is five kernels: the scan for the nearest centres (nearest.cuh), the fp64 distance to the one found,
// the minibatch ordered by centre, the update, the reassignment of starved centres. The inertia of a
// minibatch is a sum of `batch` terms in order -- 4096 dependent additions, 20 us -- and only decides whether
// another step follows, so it is taken by one block per pair beside the next step's scan, which reads nothing
// that it writes; from the kernel after that on, a fit that has stopped does nothing. At 4 pairs, batch
// 4096 and 2048 centres a step was 0.94 ms (0.84 of it fp64 distances to every centre).
__device__ __forceinline__ bool pair_active(const KmeansParams &p, const Pair &q, int t)
{
    return t < q.t_max && !p.state[q.id].stopped;
}

// Four components of a centre per lane of a warp: the fp64 centre, its 16-bit split and its bound constant.
template <bool kHalf>
__device__ __forceinline__ void store_centre(const KmeansParams &p, size_t centre, const double (&v)[4])
{
    const int lane = threadIdx.x & 31;
    uint16_t hi[4], mid[4];
    float n = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        split_component<kHalf>(v[e], hi[e], mid[e]);
        n = fmaf((float)v[e], (float)v[e], n);
    }
    n = warp_sum(n);
    const float bias = centre_bias<kHalf>(n);
    const bool fits = bias > -CUDART_INF_F;
    double2 *to = reinterpret_cast<double2 *>(p.centres64 + centre * kHeadDim + 4 * lane);
    to[0] = make_double2(v[0], v[1]);
    to[1] = make_double2(v[2], v[3]);
    auto pack = [&](const uint16_t (&h)[4]) {
        return fits ? make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16)) : make_uint2(0u, 0u);
    };
    reinterpret_cast<uint2 *>(p.centre_hi + centre * kHeadDim)[lane] = pack(hi);
    reinterpret_cast<uint2 *>(p.centre_mid + centre * kHeadDim)[lane] = pack(mid);
    if (lane == 0) p.centre_bias[centre] = bias;
}

// The centres as the start left them, their counts and the fits' state at zero. A warp per centre.
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
km_prepare_kernel(KmeansParams p)
{
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    const int u = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) p.state[q.id] = KmeansState{0.0, 0.0, 0, 0, 0, 0};
    if (u >= q.k) return;
    const double2 *from = reinterpret_cast<const double2 *>(p.centres64 + (q.cplane + u) * kHeadDim + 4 * lane);
    const double2 v0 = from[0], v1 = from[1];
    const double v[4] = {v0.x, v0.y, v1.x, v1.y};
    store_centre<kHalf>(p, q.cplane + u, v);
    if (lane == 0) p.count[q.cplane + u] = 0.0;
}

// Averaged inertia of step t and the stopping rule, one block per pair. The sum of the minibatch distances in
// order runs on one thread over shared memory that all threads filled.
__device__ __forceinline__ void km_stop_rule(const KmeansParams &p, const Pair &q, int t, double *dist_s)
{
    if (t < 0 || !pair_active(p, q, t)) return;
    const double *dist = p.dist + (size_t)q.id * p.batch;
    for (int s = threadIdx.x; s < p.batch; s += blockDim.x) dist_s[s] = dist[s];
    __syncthreads();
    if (threadIdx.x != 0) return;
    double inertia = 0.0;
#pragma unroll 16
    for (int s = 0; s < p.batch; ++s) inertia = __dadd_rn(inertia, dist_s[s]);
    KmeansState &st = p.state[q.id];
    double alpha = __ddiv_rn(__dmul_rn(2.0, (double)p.batch), __dadd_rn((double)q.N, 1.0));
    if (alpha > 1.0) alpha = 1.0;
    const double per_point = __ddiv_rn(inertia, (double)p.batch);
    const double ewa = t == 0 ? per_point
                              : __dadd_rn(__dmul_rn(st.ewa, __dsub_rn(1.0, alpha)), __dmul_rn(per_point, alpha));
    st.ewa = ewa;
    st.steps += 1;
    if (t == 0 || ewa < st.ewa_min) { st.ewa_min = ewa; st.bad = 0; }
    else if (++st.bad >= p.patience) st.stopped = 1;
}

__global__ void __launch_bounds__(kThreads)
km_last_stop_rule_kernel(KmeansParams p, int t)
{
    __shared__ double dist_s[4096];
    step_wait();
    km_stop_rule(p, pair_of(p, blockIdx.x / p.n_kv, blockIdx.x % p.n_kv), t, dist_s);
}

// Draw the minibatch and scan the centres for each point's nearest: block (256 points, pair, slice of the
// centres). Blocks of slice `assign_split` take the stopping rule of the step before instead.
template <bool kHalf>
__global__ void __launch_bounds__(kNearThreads, 2)
km_scan_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    NearSmem &sm = *reinterpret_cast<NearSmem *>(smem_raw);
    __shared__ int idx_s[kNearPoints];
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    const int slice = blockIdx.z, tid = threadIdx.x;
    if (slice == p.assign_split) {
        if (blockIdx.x == 0) km_stop_rule(p, q, t - 1, reinterpret_cast<double *>(smem_raw));
        return;
    }
    if (!pair_active(p, q, t)) return;                      // (a fit that is being stopped now may still be scanned)
    const int per = ((q.k + p.assign_split - 1) / p.assign_split + kNearTile - 1) / kNearTile * kNearTile;
    const int k_lo = min(slice * per, q.k), k_hi = min(k_lo + per, q.k);
    const int s = blockIdx.x * kNearPoints + tid;
    idx_s[tid] = km_index(km_word(p, (uint32_t)(s < p.batch ? s : 0), kTagBatch, q.stream, (uint32_t)t), q.N);
    if (slice == 0 && s < p.batch) p.idx[(size_t)q.id * p.batch + s] = idx_s[tid];
    __syncwarp();
    const uint16_t *keys = p.k_prompt + q.plane * kHeadDim;
    uint32_t a[2][8][4];
    near_load_points<kHalf>(sm, [&](int i) { return keys + (size_t)idx_s[i] * kHeadDim; }, a);
    const uint4 *hi = reinterpret_cast<const uint4 *>(p.centre_hi + q.cplane * kHeadDim);
    const uint4 *mid = reinterpret_cast<const uint4 *>(p.centre_mid + q.cplane * kHeadDim);
    const float *bias = p.centre_bias + q.cplane;
    near_scan<kHalf>(sm, a, k_lo, k_hi, [&](int stage, int base, int n) {
#pragma unroll
        for (int m = 0; m < kNearTile * 16 / kNearThreads; ++m) {
            const int e = m * kNearThreads + tid, row = e >> 4, ch = e & 15;
            if (row < n) {
                copy16_async(shared_addr(&sm.ring[stage][0][near_piece(row, ch)]), hi + (size_t)base * 16 + e);
                copy16_async(shared_addr(&sm.ring[stage][1][near_piece(row, ch)]), mid + (size_t)base * 16 + e);
            }
        }
        if (tid < kNearTile) sm.bias[stage][tid] = tid < n ? bias[base + tid] : CUDART_INF_F;
    });
    if (s < p.batch) {
        p.near_top[((size_t)q.id * p.assign_split + slice) * p.batch + s] = sm.top[tid];
        if (slice == 0) p.near_nx[(size_t)q.id * p.batch + s] = sm.nx[tid];
    }
}

// The nearest centre of each minibatch point and the fp64 distance to it: the slices' results merged, the
// candidates that the bounds leave open compared in fp64. A thread per point.
constexpr int kResolveThreads = 64;
template <bool kHalf>
__global__ void __launch_bounds__(kResolveThreads)
km_resolve_kernel(KmeansParams p, int t)
{
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    if (!pair_active(p, q, t)) return;
    const int s = blockIdx.x * kResolveThreads + threadIdx.x, lane = threadIdx.x & 31;
    const bool live = s < p.batch;
    const size_t at = (size_t)q.id * p.batch + (live ? s : 0);
    const uint4 *x = reinterpret_cast<const uint4 *>(p.k_prompt + (q.plane + (size_t)p.idx[at]) * kHeadDim);
    const double *cen = p.centres64 + q.cplane * kHeadDim;
    NearTop top = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, 0, 0};
    for (int slice = 0; slice < p.assign_split; ++slice)
        near_merge(top, p.near_top[((size_t)q.id * p.assign_split + slice) * p.batch + (live ? s : 0)]);
    const float nx = p.near_nx[at];
    bool all = !(nx <= 1e37f) || !(fabsf(top.t1) < CUDART_INF_F);
    int arg = top.i1;
    double best = CUDART_INF;
    if (!all) {
        const float bar = top.t1 + near_slack<kHalf>(nx, p.centre_bias[q.cplane + top.i1] * (1.f + 2.f * kNearErr));
        all = !(top.t3 > bar);
        if (!all) {
            best = near_exact<kHalf>(x, cen + (size_t)arg * kHeadDim);
            if (!(top.t2 > bar)) {
                const double d2 = near_exact<kHalf>(x, cen + (size_t)top.i2 * kHeadDim);
                if (d2 < best || (d2 == best && top.i2 < arg)) { best = d2; arg = top.i2; }
            }
        }
    }
    for (unsigned left = __ballot_sync(0xFFFFFFFFu, live && all); left; left &= left - 1) {
        const int l = __ffs(left) - 1;
        const uint4 *xl = reinterpret_cast<const uint4 *>(__shfl_sync(0xFFFFFFFFu, (unsigned long long)x, l));
        double d;
        const int u = near_scan_exact<kHalf>(xl, cen, q.k, d);
        if (lane == l) { best = d; arg = u; }
    }
    if (live) {
        p.label[at] = arg;
        p.dist[at] = best;
    }
}

// The minibatch ordered by (label, slot), one block per pair: two stable counting passes over the label's digits
// (kSortBits each), then where each label starts. A thread holds four consecutive entries; ranks of equal
// digits come from the warp (in order) and from counts of the warps before. (A bitonic sort of the same
// keys took 24 us.)
constexpr int kSortThreads = 1024, kSortKeys = 4096, kSortBits = 7, kSortDigits = 1 << kSortBits, kSortWarps = kSortThreads / 32;
struct SortSmem {
    uint32_t key[2][kSortKeys];                             // label << 12 | slot
    uint16_t count[kSortDigits][kSortWarps + 1];
    int scan[33];
};
__global__ void __launch_bounds__(kSortThreads)
km_sort_batch_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SortSmem &sm = *reinterpret_cast<SortSmem *>(smem_raw);
    step_wait();
    const Pair q = pair_of(p, blockIdx.x / p.n_kv, blockIdx.x % p.n_kv);
    if (!pair_active(p, q, t)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int s = tid; s < kSortKeys; s += kSortThreads)
        sm.key[0][s] = s < p.batch ? ((uint32_t)p.label[(size_t)q.id * p.batch + s] << 12) | (uint32_t)s : 0xFFFFFFFFu;
    for (int pass = 0; pass < 2; ++pass) {
        const int shift = 12 + pass * kSortBits;
        for (int e = tid; e < kSortDigits * (kSortWarps + 1); e += kSortThreads) (&sm.count[0][0])[e] = 0;
        __syncthreads();
        uint32_t key[4];
        int digit[4], rank[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {                       // the warp's 128 entries, 32 at a time in order
            key[c] = sm.key[pass][warp * 128 + c * 32 + lane];
            digit[c] = (int)((key[c] >> shift) & (kSortDigits - 1));
            const unsigned same = __match_any_sync(0xFFFFFFFFu, digit[c]);
            const int before = sm.count[digit[c]][warp];
            rank[c] = before + __popc(same & ((1u << lane) - 1u));
            __syncwarp();
            if ((same & ((1u << lane) - 1u)) == 0u) sm.count[digit[c]][warp] = (uint16_t)(before + __popc(same));
            __syncwarp();
        }
        __syncthreads();
        // exclusive prefix over (digit, warp): thread = digit * 8 + part of four warps
        {
            const int d = tid >> 3, w0 = (tid & 7) * 4;
            int n[4], sum = 0, total;
#pragma unroll
            for (int w = 0; w < 4; ++w) { n[w] = sm.count[d][w0 + w]; sum += n[w]; }
            int at = block_exclusive_scan(sum, sm.scan, total);
#pragma unroll
            for (int w = 0; w < 4; ++w) { sm.count[d][w0 + w] = (uint16_t)at; at += n[w]; }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c) sm.key[pass ^ 1][sm.count[digit[c]][warp] + rank[c]] = key[c];
        __syncthreads();
    }
    const int32_t *idx = p.idx + (size_t)q.id * p.batch;
    int32_t *start = p.start + (size_t)q.id * (p.k_max + 1);
    for (int s = tid; s < kSortKeys; s += kSortThreads) {
        const uint32_t key = sm.key[0][s];
        const int label = min((int)(key >> 12), q.k);       // (the padding sorts behind every label)
        const int prev = s > 0 ? min((int)(sm.key[0][s - 1] >> 12), q.k) : -1;
        for (int u = prev + 1; u <= label; ++u) start[u] = s;
        if (s == kSortKeys - 1)
            for (int u = label + 1; u <= q.k; ++u) start[u] = kSortKeys;
        if (s < p.batch) p.sorted[(size_t)q.id * kSortKeys + s] = idx[key & 4095u];
    }
}

// Cumulative-count update, a warp per centre (four dimensions per lane): the centre's new points are added in
// minibatch order, eight rows requested at a time; c <- (c * count + sum) / (count + n).
template <bool kHalf>
__global__ void __launch_bounds__(128)
km_batch_update_kernel(KmeansParams p, int t)
{
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    if (!pair_active(p, q, t)) return;
    const int u = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (u >= q.k) return;
    const int32_t *start = p.start + (size_t)q.id * (p.k_max + 1);
    const int lo = start[u], hi = start[u + 1];
    if (lo == hi) return;
    const int32_t *point = p.sorted + (size_t)q.id * kSortKeys;
    const uint2 *keys = reinterpret_cast<const uint2 *>(p.k_prompt + q.plane * kHeadDim) + lane;
    const double count = p.count[q.cplane + u];
    const double2 *from = reinterpret_cast<const double2 *>(p.centres64 + (q.cplane + u) * kHeadDim + 4 * lane);
    const double2 c0 = from[0], c1 = from[1];
    double sum[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i0 = lo; i0 < hi; i0 += 8) {
        uint2 w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = __ldg(keys + (size_t)point[min(i0 + i, hi - 1)] * 32);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i0 + i >= hi) break;
            sum[0] = __dadd_rn(sum[0], (double)elem_lo<kHalf>(w[i].x));
            sum[1] = __dadd_rn(sum[1], (double)elem_hi<kHalf>(w[i].x));
            sum[2] = __dadd_rn(sum[2], (double)elem_lo<kHalf>(w[i].y));
            sum[3] = __dadd_rn(sum[3], (double)elem_hi<kHalf>(w[i].y));
        }
    }
    const double grown = __dadd_rn(count, (double)(hi - lo)), c[4] = {c0.x, c0.y, c1.x, c1.y};
    double v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = __ddiv_rn(__dadd_rn(__dmul_rn(c[e], count), sum[e]), grown);
    store_centre<kHalf>(p, q.cplane + u, v);
    if (lane == 0) p.count[q.cplane + u] = grown;
}

// Reassignment of starved centres, one block per pair.
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
km_reassign_kernel(KmeansParams p, int t)
{
    extern __shared__ int32_t slots[];                      // slots[batch], then move_centre[batch / 2]
    __shared__ int n_move_s;
    __shared__ double cmin_s[kThreads / 32], cmax_s[kThreads / 32];
    step_wait();
    const Pair q = pair_of(p, blockIdx.x, blockIdx.y);
    if (!(p.ratio > 0.0) || !pair_active(p, q, t)) return;
    const int tid = threadIdx.x;
    int32_t *move_centre = slots + p.batch;
    double *count = p.count + q.cplane;
    {
        double cmin = INFINITY, cmax = 0.0;                 // smallest and largest count: any order gives the same
        for (int u = tid; u < q.k; u += kThreads) {
            const double v = count[u];
            if (v < cmin) cmin = v;
            if (v > cmax) cmax = v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double a = __shfl_xor_sync(0xffffffffu, cmin, o), b = __shfl_xor_sync(0xffffffffu, cmax, o);
            if (a < cmin) cmin = a;
            if (b > cmax) cmax = b;
        }
        if ((tid & 31) == 0) { cmin_s[tid >> 5] = cmin; cmax_s[tid >> 5] = cmax; }
    }
    __syncthreads();
    if (tid == 0) {
        int n_move = 0;
        double cmin = INFINITY, cmax = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) {
            if (cmin_s[w] < cmin) cmin = cmin_s[w];
            if (cmax_s[w] > cmax) cmax = cmax_s[w];
        }
        const long long period = 10 + (long long)floor(cmin);
        if (((long long)t + 1) % period == 0) {
            const double thr = __dmul_rn(p.ratio, cmax);
            const int cap = p.batch / 2;
            double keep_min = INFINITY;
            for (int u = 0; u < q.k; ++u) {
                const double v = count[u];
                if (v < thr && n_move < cap) move_centre[n_move++] = u;
                else if (v < keep_min) keep_min = v;
            }
            if (n_move > 0) {
                for (int s = 0; s < p.batch; ++s) slots[s] = s;
                for (int i = 0; i < n_move; ++i) {
                    const int r = i + km_index(km_word(p, (uint32_t)i, kTagMove, q.stream, (uint32_t)t), p.batch - i);
                    const int tmp = slots[i];
                    slots[i] = slots[r];
                    slots[r] = tmp;
                }
                for (int i = 0; i < n_move; ++i) count[move_centre[i]] = keep_min;
            }
        }
        n_move_s = n_move;
    }
    __syncthreads();
    const int32_t *idx = p.idx + (size_t)q.id * p.batch;
    for (int i = tid >> 5; i < n_move_s; i += kThreads / 32) {   // the moved centres jump onto minibatch points
        const uint2 w = reinterpret_cast<const uint2 *>(p.k_prompt + (q.plane + (size_t)idx[slots[i]]) * kHeadDim)[tid & 31];
        const double v[4] = {(double)elem_lo<kHalf>(w.x), (double)elem_hi<kHalf>(w.x), (double)elem_lo<kHalf>(w.y), (double)elem_hi<kHalf>(w.y)};
        store_centre<kHalf>(p, q.cplane + move_centre[i], v);
    }
}

// How many fits still have steps to run after step t (one block; the host reads it now and then
// and stops enqueuing steps once it is zero).
__global__ void __launch_bounds__(kThreads)
km_count_active_kernel(KmeansParams p, int t)
{
    __shared__ int n_s;
    if (threadIdx.x == 0) n_s = 0;
    __syncthreads();
    const int pairs = p.n_seqs * p.n_kv;
    int n = 0;
    for (int i = threadIdx.x; i < pairs; i += kThreads) {
        const int b = i % p.n_seqs;                         // state is indexed j * n_seqs + b
        n += (t + 1 < p.seq_t_max[b] && !p.state[i].stopped) ? 1 : 0;
    }
    if (n) atomicAdd(&n_s, n);
    __syncthreads();
    if (threadIdx.x == 0) *p.active = n_s;
}

__global__ void __launch_bounds__(kThreads)
km_finish_kernel(KmeansParams p)
{
    const Pair q = pair_of(p, blockIdx.y, blockIdx.z);
    const int e = blockIdx.x * kThreads + threadIdx.x;
    if (e < q.k * kHeadDim) p.centres_out[q.cplane * kHeadDim + e] = __double2float_rn(p.centres64[q.cplane * kHeadDim + e]);
    if (e == 0 && p.steps_out) p.steps_out[q.id] = p.state[q.id].steps;
}

template <bool kHalf>
cudaError_t run_fit(const KmeansParams &p, cudaStream_t s)
{
    const int B = p.n_seqs, H = p.n_kv, pairs = B * H;
    cudaError_t err;
#define KM_CHECK() if ((err = cudaGetLastError()) != cudaSuccess) return err
    static std::atomic<unsigned long long> sample_done;
    if ((err = ensure_dynamic_smem((const void *)km_sample_kernel, (int)sample_smem(kMaxSumBlocks * kSumBlock), sample_done)) != cudaSuccess) return err;
    if ((err = launch_step(km_sample_kernel, dim3(B, H), dim3(kSampleThreads), sample_smem(p.n_init_max), s, p)) != cudaSuccess) return err;
    const dim3 dist_grid((p.n_init_max + kSumBlock - 1) / kSumBlock, (p.trials_max + kDistTrials - 1) / kDistTrials, pairs);
    const size_t draw_smem = sizeof(double) * ((size_t)p.n_init_max + 2 * kMaxSumBlocks);
    if ((err = cudaFuncSetAttribute(km_accept_kernel<kHalf>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)draw_smem)) != cudaSuccess)
        return err;
    for (int c = 0; c < p.k_max; ++c) {
        km_candidate_dist_kernel<kHalf><<<dist_grid, kDistThreads, 0, s>>>(p, c);
        KM_CHECK();
        km_accept_kernel<kHalf><<<dim3(B, H), kAcceptThreads, draw_smem, s>>>(p, c);     // ... and the trial points of centre c + 1
        KM_CHECK();
    }
    const dim3 threads(kThreads);
    if ((err = launch_step(km_prepare_kernel<kHalf>, dim3((p.k_max + kThreads / 32 - 1) / (kThreads / 32), pairs), threads, 0, s, p)) != cudaSuccess) return err;
    static std::atomic<unsigned long long> scan_done, sort_done;
    if ((err = ensure_dynamic_smem((const void *)km_scan_kernel<kHalf>, (int)sizeof(NearSmem), scan_done)) != cudaSuccess) return err;
    if ((err = ensure_dynamic_smem((const void *)km_sort_batch_kernel, (int)sizeof(SortSmem), sort_done)) != cudaSuccess) return err;
    const size_t move_smem = sizeof(int32_t) * ((size_t)p.batch + (size_t)p.batch / 2 + 1);
    const dim3 scan_grid((p.batch + kNearPoints - 1) / kNearPoints, pairs, p.assign_split + 1);
    const dim3 resolve_grid((p.batch + kResolveThreads - 1) / kResolveThreads, pairs);
    int t = 0;
    for (; t < p.t_max_max; ++t) {
        if ((err = launch_step(km_scan_kernel<kHalf>, scan_grid, dim3(kNearThreads), sizeof(NearSmem), s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_resolve_kernel<kHalf>, resolve_grid, dim3(kResolveThreads), 0, s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_sort_batch_kernel, dim3(pairs), dim3(kSortThreads), sizeof(SortSmem), s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_batch_update_kernel<kHalf>, dim3((p.k_max + 3) / 4, pairs), dim3(128), 0, s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_reassign_kernel<kHalf>, dim3(B, H), threads, move_smem, s, p, t)) != cudaSuccess) return err;
        if (!p.no_host_poll && (t + 1) % kPollEvery == 0 && t + 1 < p.t_max_max) {
            // most fits stop long before the step limit: ask the device how many are still running
            // (the copy into pageable memory returns when it has completed)
            int active = 1;
            km_count_active_kernel<<<1, kThreads, 0, s>>>(p, t);
            KM_CHECK();
            if ((err = cudaMemcpyAsync(&active, p.active, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return err;
            if ((err = cudaStreamSynchronize(s)) != cudaSuccess) return err;
            if (active == 0) { ++t; break; }
        }
    }
    if ((err = launch_step(km_last_stop_rule_kernel, dim3(pairs), threads, 0, s, p, t - 1)) != cudaSuccess) return err;   // counts the last step
    km_finish_kernel<<<dim3((p.k_max * kHeadDim + kThreads - 1) / kThreads, B, H), kThreads, 0, s>>>(p);
    KM_CHECK();
#undef KM_CHECK
    return cudaSuccess;
}

}  // namespace

namespace {
__global__ void __launch_bounds__(kKmTableChunk + 32)
km_tables_kernel(const __grid_constant__ KmTableChunk c, int64_t *row_off, int64_t *centre_off, int32_t *n_init,
                 int32_t *trials, int32_t *t_max)
{
    const int i = threadIdx.x;
    if (i <= c.n) {
        row_off[c.first + i] = c.row_off[i];
        centre_off[c.first + i] = c.centre_off[i];
    }
    if (i < c.n) {
        n_init[c.first + i] = c.n_init[i];
        trials[c.first + i] = c.trials[i];
        t_max[c.first + i] = c.t_max[i];
    }
}
}  // namespace

cudaError_t launch_kmeans_tables(const KmTableChunk &c, int64_t *row_off, int64_t *centre_off, int32_t *n_init,
                                 int32_t *trials, int32_t *t_max, cudaStream_t s)
{
    km_tables_kernel<<<1, kKmTableChunk + 32, 0, s>>>(c, row_off, centre_off, n_init, trials, t_max);
    return cudaGetLastError();
}

cudaError_t launch_kmeans_fit(const KmeansParams &p, cudaStream_t s)
{
    return p.elem ? run_fit<true>(p, s) : run_fit<false>(p, s);
}

}  // namespace santapp
