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
    if (tid == 0) p.chosen[q.cplane + (size_t)c] = p.pick[(size_t)q.id * p.trials_max + best];
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

// The greedy start as one kernel: a cluster of blocks per pair that keeps the sample in shared memory (for samples
// of at most kStartRows rows per block; the two kernels per centre above take larger ones).
//
// Only the winning trial's distances are needed in fp64. A trial lowers the potential by the sum over the points
// of what it takes off their nearest-centre distance, and the products of the rows with the trial points give every
// such gain within a bound (select_rows.cuh). Per centre the cluster's blocks
//   1. multiply their rows with the trial points on tensor cores, mark the points that a trial may lower, add up
//      each trial's largest and smallest possible gain, and send one another the sums;
//   2. take the trial whose smallest gain exceeds every other's largest; if there is none, the potentials are
//      summed in fp64 for all trials (a few centres in two thousand; trials that drew the same point do not count);
//   3. evaluate the winner's marked points in fp64 (a handful, after the first hundred centres), lower the
//      distances, renew the running sums of the blocks of the sums they lie in, and send those blocks' sums;
//   4. add up the blocks and draw the next trial points: the block that owns a drawn point sends its row to all.
// Bound by the chain of a centre, 12300 cycles (6.4 us) of 12288 points and nine trials: 4000 for the marks (1500 of them products at the
// tensor cores' rate, the rest their operands, the look at the results and the slowest warp) and the gains' sums, 2000 for the gains'
// message and the winner, 3600 until the slowest block's distances and running sums (128 terms in order, 11 cycles each) are
// there, 1100 for the blocks' sums (96 terms), 1600 for the draws and their rows. Messages are stores that count their bytes on an
// mbarrier of the block they go to, 700 cycles; with cluster barriers behind remote stores, three of 1900 cycles, all of
// a block's threads waiting for the slowest block's, and a distance summed in order by one lane (1100 cycles a point), a
// centre took 8.2 us. Twelve warps, four tiles each, so that three warps a scheduler overlap operands, products and
// marks (eight warps: 6.9 us a centre; sixteen: 6.6, with a barrier and the slowest warp of more): fits of 32768 keys to 2048, 256 and 64
// centres 22.1 -> 18.2, 6.35 -> 5.10 and 4.63 -> 3.81 ms with the steps below. The operands wait in tensor
// memory: read from shared memory they are as long on their way as the products take. (tcgen05 itself: sixteen
// columns take as long as 128, 9 us a centre.) The two kernels per centre took 38 us, 24 of them fp64 distances of
// every point to every trial.
constexpr int kStartThreads = 384, kStartWarps = kStartThreads / 32;
constexpr int kStartBlocks = 6;          // blocks of the sums per thread block: 768 rows of 256 bytes
constexpr int kStartRows = kStartBlocks * kSumBlock;
constexpr int kStartTmp = 4;             // warps that sum potentials
// The messages of a centre. A block that owns sums sends them when it has all gains, so nobody starts the next centre before; one that owns
// none is not waited for, and the next centre's gains can reach it ahead of the last of this one's: gains have a barrier for each parity of
// the centre (those of the centre after the next follow the gains that this block sends for the next).
// Potentials lie in global memory; kPotentials counts the warps of the cluster that have written theirs.
enum { kGains, kSums = 2, kDraws, kPotentials, kMessages };
constexpr int kStartMaxCluster = 16, kStartSums = kStartBlocks * kStartMaxCluster;
constexpr int kStartTrials = 11;         // 2 + floor(ln k) for every k with a sample of at most 16 * kStartRows: k <= 12288, ln k < 10
static_assert(kStartTrials <= kStartWarps, "a warp per draw");
static_assert(kStartMaxCluster * kStartRows < 22026, "e^10: from there on a centre has more trials");

struct StartDraw {                       // a drawn trial point: squared norm, index in the sample, unit (elem_unit of its row)
    float norm;
    int pick, unit, pad;
};
struct StartSmem {
    alignas(16) uint4 rows[kStartRows * 16];                // 16-byte pieces XOR-swizzled (near_piece)
    uint4 trial[kStartTrials * 16];
    double closest[kStartRows];
    double run[kStartRows];                                 // running sums of the distances inside each block of the sums
    double tmp[kStartTmp][kSumBlock];
    double raw[kStartSums];                                 // sums of all the pair's blocks
    double pre[kStartSums];                                 // ... and their running sums
    float norm[kStartRows];                                 // squared norms
    float bar[kStartRows];                                  // norm * (1 - error) - nearest-centre distance; infinite where no centre is nearer
    float2 gain[2][kStartMaxCluster][kStartTrials];         // (smallest, largest) gain of a trial over each block's points, by the centre's parity
    float own_gain[2][kStartTrials][2];                     // of this block, by the centre's parity
    alignas(16) StartDraw draw[2][kStartTrials];            // the trial points, by the centre's parity
    uint64_t arrived[kMessages];                            // mbarriers: every block's gains, block sums, trial points, potentials
    uint32_t touched[kStartBlocks];                         // trials with a marked point in the block
    uint32_t tmem;
    int failed;                                             // a wait ran out (never expected)
    uint16_t mask[kStartRows];                              // trials that may lower the point's distance
    int8_t unit[kStartRows];                                // every value of the row is a multiple of 2^unit; -128: not known
    uint8_t list[kStartWarps][kSumBlock];                   // marked points of a warp's block
};
static_assert(sizeof(StartSmem) <= 227 * 1024, "shared memory of one block");

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t in_block(uint32_t addr, uint32_t rank)      // the same shared-memory address in another block
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Every thread of the cluster; the warp has to be whole (it is brought together first).
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    __syncwarp();
}

// Messages between the blocks of a cluster: stores into another block's shared memory that count their bytes on an mbarrier there.
__device__ __forceinline__ void send2(uint32_t to, uint32_t bar, float x, float y)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(to), "f"(x), "f"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void send_double(uint32_t to, uint32_t bar, double x)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(to), "d"(x), "r"(bar) : "memory");
}
__device__ __forceinline__ void send4(uint32_t to, uint32_t bar, uint4 v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(to), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
// Arrival at a barrier of another block of the cluster, behind what the warp's lanes have written.
__device__ __forceinline__ void arrive_at(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void expect_bytes(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(shared_addr(bar)), "r"(bytes) : "memory");
}

// The exponent of a 16-bit value's lowest set bit; 127 for zero, -128 where it is -128 or below.
template <bool kHalf>
__device__ __forceinline__ int elem_unit(uint32_t v)
{
    constexpr int kMan = kHalf ? 10 : 7, kLow = kHalf ? -24 : -133;         // mantissa bits, exponent of the smallest subnormal
    const int e = (int)((v & 0x7FFFu) >> kMan), m = (int)(v & ((1u << kMan) - 1u)) | (e > 0 ? 1 << kMan : 0);
    return m == 0 ? 127 : max(kLow + max(e, 1) - 1 + __ffs(m) - 1, -128);
}
// The smallest of a row's, by a warp.
template <bool kHalf>
__device__ __forceinline__ int row_unit(const uint4 *rows, int i)
{
    const int lane = threadIdx.x & 31;
    const uint2 w = reinterpret_cast<const uint2 *>(rows + near_piece(i, lane >> 1))[lane & 1];
    return __reduce_min_sync(0xFFFFFFFFu, min(min(elem_unit<kHalf>(w.x & 0xFFFFu), elem_unit<kHalf>(w.x >> 16)),
                                              min(elem_unit<kHalf>(w.y & 0xFFFFu), elem_unit<kHalf>(w.y >> 16))));
}
// Squared norm of a row by a warp (an fp32 sum; every lane gets it).
template <bool kHalf>
__device__ __forceinline__ float row_norm(const uint4 *rows, int i)
{
    const int lane = threadIdx.x & 31;
    const uint2 w = reinterpret_cast<const uint2 *>(rows + near_piece(i, lane >> 1))[lane & 1];
    const float a = elem_lo<kHalf>(w.x), b = elem_hi<kHalf>(w.x), c = elem_lo<kHalf>(w.y), d = elem_hi<kHalf>(w.y);
    return warp_sum(fmaf(a, a, b * b) + fmaf(c, c, d * d));
}

// src[from .. cnt) added in order to w, one lane; dst gets the running sums (dst may be src). Eight terms are loaded while
// the eight before them are added.
__device__ __forceinline__ double run_sums(const double *src, double *dst, int from, int cnt, double w)
{
    int u = from;
    for (; u < cnt && (u & 7); ++u) { w = __dadd_rn(w, src[u]); dst[u] = w; }
    if (u + 8 <= cnt) {
        double t[8];
#pragma unroll
        for (int e = 0; e < 8; e += 2) *reinterpret_cast<double2 *>(&t[e]) = *reinterpret_cast<const double2 *>(src + u + e);
        for (; u + 8 <= cnt; u += 8) {
            double n[8];
            const int nx = u + 16 <= cnt ? u + 8 : u;
#pragma unroll
            for (int e = 0; e < 8; e += 2) *reinterpret_cast<double2 *>(&n[e]) = *reinterpret_cast<const double2 *>(src + nx + e);
#pragma unroll
            for (int e = 0; e < 8; ++e) { w = __dadd_rn(w, t[e]); t[e] = w; }
#pragma unroll
            for (int e = 0; e < 8; e += 2) *reinterpret_cast<double2 *>(dst + u + e) = *reinterpret_cast<const double2 *>(&t[e]);
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] = n[e];
        }
    }
    for (; u < cnt; ++u) { w = __dadd_rn(w, src[u]); dst[u] = w; }
    return w;
}

// The defining distance of two rows, one lane.
template <bool kHalf>
__device__ __forceinline__ double start_dist(const uint4 *rows, int i, const uint4 *trial, int l)
{
    double s = 0.0;
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
        const uint4 x4 = rows[near_piece(i, c)], y4 = trial[near_piece(l, c)];
        const uint32_t x[4] = {x4.x, x4.y, x4.z, x4.w}, y[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double e0 = __dsub_rn((double)elem_lo<kHalf>(x[t]), (double)elem_lo<kHalf>(y[t]));
            const double e1 = __dsub_rn((double)elem_hi<kHalf>(x[t]), (double)elem_hi<kHalf>(y[t]));
            s = __dadd_rn(s, __dmul_rn(e0, e0));
            s = __dadd_rn(s, __dmul_rn(e1, e1));
        }
    }
    return s;
}
// Eight consecutive values as doubles.
template <bool kHalf>
__device__ __forceinline__ void widen8(const uint4 &w4, double (&v)[8])
{
    const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        v[2 * t] = (double)elem_lo<kHalf>(w[t]);
        v[2 * t + 1] = (double)elem_hi<kHalf>(w[t]);
    }
}
// An eighth of that distance in any order: pieces `part` and `part + 8` of row i against a trial point's, y.
template <bool kHalf>
__device__ __forceinline__ double start_dist_part(const uint4 *rows, int i, int part, const double (&y)[2][8])
{
    double s[2] = {0.0, 0.0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        double x[8];
        widen8<kHalf>(rows[near_piece(i, part + 8 * h)], x);
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const double e = x[t] - y[h][t];
            s[h] = fma(e, e, s[h]);
        }
    }
    return s[0] + s[1];
}
// A lane of every eight gets the sum of the eight lanes' parts (all eight do).
__device__ __forceinline__ double sum_parts(double s)
{
    s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
    s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
    return s + __shfl_xor_sync(0xFFFFFFFFu, s, 4);
}

template <bool kHalf>
__global__ void __launch_bounds__(kStartThreads, 1)
km_start_kernel(KmeansParams p)
{
    extern __shared__ __align__(128) unsigned char start_smem[];
    StartSmem &sm = *reinterpret_cast<StartSmem *>(start_smem);
    constexpr float kPairErr = 0.5f * kDistErr;             // times the sum of the two squared norms, plus kUnderflow
    // The rows as mma.sync's first operands (a word per lane, tile of 16 rows, step of 16 values: 32 columns a tile) in tensor memory,
    // a warp's tiles m = warp, warp + kStartWarps, ... behind one another, three warps to a quarter of the lanes.
    constexpr int kTiles = kStartRows / 16 / kStartWarps, kTmemCols = 512;
    static_assert(kStartWarps / 4 * kTiles * 32 <= kTmemCols, "operands in tensor memory");
    const int n_blk = (int)cluster_size(), rank = (int)cluster_rank();
    const int pair = blockIdx.x / n_blk, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, c4 = lane & 3;
    const Pair q = pair_of(p, pair / p.n_kv, pair % p.n_kv);
    const int nb = (q.n_init + kSumBlock - 1) / kSumBlock;  // blocks of the sums; this thread block's are [b0, b0 + mb)
    const int per = (nb + n_blk - 1) / n_blk, b0 = min(rank * per, nb), mb = min(per, nb - b0);
    const int row0 = b0 * kSumBlock, n_rows = max(min(q.n_init - row0, mb * kSumBlock), 0);
    const int32_t *perm = p.perm + q.plane;
    const uint4 *keys = reinterpret_cast<const uint4 *>(p.k_prompt + q.plane * kHeadDim);
    const int n_part = (p.n_init_max + kSumBlock - 1) / kSumBlock;
    double *part = p.part + (size_t)q.id * p.trials_max * n_part;       // [trial][n_part] block sums, where all trials are summed

    // ---- the block's rows; the first centre as the only trial point ----
    for (int e = tid; e < n_rows * 16; e += kStartThreads)
        copy16_async(shared_addr(&sm.rows[near_piece(e >> 4, e & 15)]), keys + (size_t)perm[row0 + (e >> 4)] * 16 + (e & 15));
    const int first = p.pick[(size_t)q.id * p.trials_max];
    if (tid == 0) {
        sm.failed = 0;
        for (int t = 0; t < kMessages; ++t)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(shared_addr(&sm.arrived[t])), "r"(t == kPotentials ? n_blk * kStartTmp : 1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(shared_addr(&sm.tmem)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    copy_async_wait();
    for (int e = n_rows * 16 + tid; e < mb * kSumBlock * 16; e += kStartThreads) sm.rows[near_piece(e >> 4, e & 15)] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int tiles = mb * (kSumBlock / 16);
    const uint32_t operands = sm.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * kTiles * 32);
    for (int n = 0; warp + kStartWarps * n < tiles; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t f[4];
                ldmatrix4(f, shared_addr(&sm.rows[near_piece((warp + kStartWarps * n) * 16 + (lane & 15), 8 * h + 2 * e + (lane >> 4))]));
                w[4 * e] = f[0]; w[4 * e + 1] = f[1]; w[4 * e + 2] = f[2]; w[4 * e + 3] = f[3];
            }
            tc_st16(operands + (uint32_t)(32 * n + 16 * h), w);
        }
    for (int i = warp; i < mb * kSumBlock; i += kStartWarps) {
        const float n = i < n_rows ? row_norm<kHalf>(sm.rows, i) : 0.f;
        const int unit = i < n_rows ? row_unit<kHalf>(sm.rows, i) : 0;
        if (lane == 0) {
            sm.norm[i] = n;
            sm.unit[i] = (int8_t)unit;
            sm.closest[i] = i < n_rows ? CUDART_INF : 0.0;
            sm.bar[i] = i < n_rows ? 0.f : CUDART_INF_F;    // (set with the first distances)
            sm.mask[i] = i < n_rows ? 1 : 0;
        }
    }
    if (warp == 0) {
        const uint4 piece = __ldg(keys + (size_t)perm[first] * 16 + (lane & 15));
        if (lane < 16) sm.trial[near_piece(0, lane)] = piece;
        const uint32_t w[4] = {piece.x, piece.y, piece.z, piece.w};
        int unit = 127;
#pragma unroll
        for (int t = 0; t < 4; ++t) unit = min(unit, min(elem_unit<kHalf>(w[t] & 0xFFFFu), elem_unit<kHalf>(w[t] >> 16)));
        unit = __reduce_min_sync(0xFFFFFFFFu, unit);
        if (lane == 0) { sm.draw[0][0].unit = unit; sm.draw[0][0].pick = first; }
    }
    if (tid < kStartBlocks) sm.touched[tid] = tid < mb ? 1u : 0u;
    for (int e = tid; e < 2 * kStartMaxCluster * kStartTrials; e += kStartThreads) sm.gain[0][0][e] = make_float2(0.f, 0.f);
    if (tid < 4 * kStartTrials) sm.own_gain[0][0][tid] = 0.f;
    cluster_barrier();                                      // every block of the cluster runs: its shared memory may be written

    // Where a wait runs out the block's later ones return at once, and the block leaves the loop with the centre; what its warps decide
    // until then may differ, so between here and there stands no wait without a limit but the block's own barriers.
    auto await = [&](int what, uint32_t parity) {
        if (!*reinterpret_cast<volatile int *>(&sm.failed) && !tc_wait<true>(shared_addr(&sm.arrived[what]), parity)) sm.failed = 1;
        __syncwarp();
    };
    // a thread sends one trial's gains to one block
    const int gain_of = tid % q.L, gain_to = tid / q.L;
    const uint32_t gain_at = in_block(shared_addr(&sm.gain[0][rank][gain_of]), min(gain_to, n_blk - 1));
    const uint32_t gain_bar = in_block(shared_addr(&sm.arrived[kGains]), min(gain_to, n_blk - 1));
    uint32_t summed = 0u;                                   // centres whose potentials were summed
    float slack = 0.f;                                      // rounding of the sums that define the potentials
    for (int c = 0; c < q.k; ++c) {
        const int L = c == 0 ? 1 : q.L, par = c & 1;
        int best = 0;
        if (tid == 0) {                                     // the centre's messages to come (the ones before have all been waited for)
            if (c > 0) expect_bytes(&sm.arrived[kGains + par], (uint32_t)(n_blk * L * sizeof(float2)));
            if (c + 1 < q.k) {
                expect_bytes(&sm.arrived[kSums], (uint32_t)(nb * sizeof(double)));
                expect_bytes(&sm.arrived[kDraws], (uint32_t)(q.L * (kHeadDim * 2 + sizeof(StartDraw))));
            }
        }
        if (c > 0) {
            // ---- 1. which points a trial may lower, and by how much ----
            uint32_t bf[2][8][2];                           // the trial points as MMA columns (two groups of eight)
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int t = min(n * 8 + (lane & 7), L - 1);
#pragma unroll
                for (int s2 = 0; s2 < 4; ++s2) {
                    uint32_t r[4];
                    ldmatrix4(r, shared_addr(&sm.trial[near_piece(t, 4 * s2 + (lane >> 3))]));
                    bf[n][2 * s2][0] = r[0]; bf[n][2 * s2][1] = r[1]; bf[n][2 * s2 + 1][0] = r[2]; bf[n][2 * s2 + 1][1] = r[3];
                }
            }
            float ny[4], err[4], lo[4], hi[4];              // the thread's columns: 2 c4, 2 c4 + 1, 8 + 2 c4, 9 + 2 c4
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int t = (v >> 1) * 8 + 2 * c4 + (v & 1);
                const float n = t < L ? sm.draw[par][t].norm : 0.f;
                // (a column that is no trial is never marked; of a norm that fp32 does not hold the product decides nothing)
                ny[v] = t >= L ? CUDART_INF_F : (n <= 1e37f ? n * (1.f - kPairErr) : -CUDART_INF_F);
                err[v] = 2.f * kPairErr * n;
                lo[v] = hi[v] = 0.f;
            }
            for (int n = 0; warp + kStartWarps * n < tiles; ++n) {
                const int i0 = (warp + kStartWarps * n) * 16;
                float acc[2][4] = {};
                uint32_t a[32];
                tc_ld32(operands + (uint32_t)(32 * n), a);
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    mma_rows<kHalf>(acc[0], a[4 * s], a[4 * s + 1], a[4 * s + 2], a[4 * s + 3], bf[0][s][0], bf[0][s][1]);
                    if (L > 8) mma_rows<kHalf>(acc[1], a[4 * s], a[4 * s + 1], a[4 * s + 2], a[4 * s + 3], bf[1][s][0], bf[1][s][1]);
                }
                uint32_t bits[2];
                float val[2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float bar = sm.bar[i0 + g + 8 * h];
                    bits[h] = 0u;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        val[h][v] = fmaf(-2.f, acc[v >> 1][2 * h + (v & 1)], bar + ny[v]);
                        // (a column that is no trial beside a row without a bound: plus and minus infinity, not a number)
                        const int t = (v >> 1) * 8 + 2 * c4 + (v & 1);
                        if (!(val[h][v] > kUnderflow) && t < L) bits[h] |= 1u << t;
                    }
                    if (!(bar < CUDART_INF_F)) bits[h] = 0u;         // a centre, or past the end of the sample
                }
                if (__any_sync(0xFFFFFFFFu, (bits[0] | bits[1]) != 0u)) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float e = fmaf(2.f * kPairErr, sm.norm[i0 + g + 8 * h], kUnderflow);
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            if ((bits[h] >> ((v >> 1) * 8 + 2 * c4 + (v & 1))) & 1u) {
                                hi[v] += kUnderflow - val[h][v];
                                lo[v] += fmaxf(-val[h][v] - (e + err[v]), 0.f);
                            }
                        bits[h] |= __shfl_xor_sync(0xFFFFFFFFu, bits[h], 1);
                        bits[h] |= __shfl_xor_sync(0xFFFFFFFFu, bits[h], 2);
                    }
                    const uint32_t any = __reduce_or_sync(0xFFFFFFFFu, bits[0] | bits[1]);
                    if (lane == 0) atomicOr(&sm.touched[i0 / kSumBlock], any);
                }
                if (c4 < 2) sm.mask[i0 + g + 8 * c4] = (uint16_t)(c4 ? bits[1] : bits[0]);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {                   // (most columns have no marked point in the warp's rows)
                if (!__any_sync(0xFFFFFFFFu, hi[v] != 0.f)) continue;
#pragma unroll
                for (int o = 4; o <= 16; o <<= 1) {
                    lo[v] += __shfl_xor_sync(0xFFFFFFFFu, lo[v], o);
                    hi[v] += __shfl_xor_sync(0xFFFFFFFFu, hi[v], o);
                }
                const int t = (v >> 1) * 8 + 2 * c4 + (v & 1);
                if (g == 0 && t < L && hi[v] != 0.f) {      // (the order of these sums is covered by the 1e-5 below)
                    atomicAdd(&sm.own_gain[par][t][0], lo[v]);
                    atomicAdd(&sm.own_gain[par][t][1], hi[v]);
                }
            }
            __syncthreads();
            if (gain_to < n_blk) send2(gain_at + (uint32_t)(par * sizeof(sm.gain[0])), gain_bar + (uint32_t)(par * sizeof(uint64_t)), sm.own_gain[par][gain_of][0], sm.own_gain[par][gain_of][1]);
            const int mine = sm.draw[par][min(lane, L - 1)].pick;
            await(kGains + par, (uint32_t)((c - 1) >> 1) & 1u);
            // ---- 2. the winner ----
            {
                // every warp for itself; 1e-5: rounding of the fp32 sums; 1e-11: of the fp64 sums that define the potentials
                float gl = 0.f, gh = 0.f;
#pragma unroll
                for (int r = 0; r < kStartMaxCluster / 2; ++r) {     // half the blocks each half of the warp (zero past the cluster's)
                    const float2 v = sm.gain[par][(lane & 16) / 2 + r][min(lane & 15, L - 1)];
                    gl += v.x;
                    gh += v.y;
                }
                gl += __shfl_xor_sync(0xFFFFFFFFu, gl, 16);
                gh += __shfl_xor_sync(0xFFFFFFFFu, gh, 16);
                gl = lane < L ? gl * (1.f - 1e-5f) - slack : -CUDART_INF_F;
                gh = gh * (1.f + 1e-5f);
                const float top = warp_max(gl);
                const unsigned at = __ballot_sync(0xFFFFFFFFu, lane < L && gl == top);
                best = at ? __ffs(at) - 1 : 0;              // (gains that do not compare leave the first trial)
                const int its = __shfl_sync(0xFFFFFFFFu, mine, best);
                const bool open = lane < L && !(gh < top) && mine != its;
                if (__any_sync(0xFFFFFFFFu, open)) {
                    // all potentials in fp64: each block of the sums in order, then the blocks in order
                    for (int v = warp; warp < kStartTmp && v < L * mb; v += kStartTmp) {
                        const int l = v / mb, blk = v - l * mb, base = blk * kSumBlock;
                        double w = sm.raw[b0 + blk];
                        if ((sm.touched[blk] >> l) & 1u) {
                            __syncwarp();
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int i = base + e * 32 + lane;
                                double t = sm.closest[i];
                                if ((sm.mask[i] >> l) & 1) {
                                    const double d = start_dist<kHalf>(sm.rows, i, sm.trial, l);
                                    if (d < t) t = d;
                                }
                                sm.tmp[warp][e * 32 + lane] = t;
                            }
                            __syncwarp();
                            if (lane == 0) w = run_sums(sm.tmp[warp], sm.tmp[warp], 0, min(kSumBlock, n_rows - base), 0.0);
                        }
                        if (lane == 0) part[(size_t)l * n_part + b0 + blk] = w;
                    }
                    __syncwarp();
                    if (warp < kStartTmp && lane < n_blk) arrive_at(in_block(shared_addr(&sm.arrived[kPotentials]), lane));
                    await(kPotentials, summed++ & 1u);      // (the same decision in every warp of the cluster)
                    double pot = 0.0;
                    if (lane < L)
#pragma unroll 8
                        for (int blk = 0; blk < nb; ++blk) pot = __dadd_rn(pot, __ldcg(part + (size_t)lane * n_part + blk));
                    best = 0;
                    double low = __shfl_sync(0xFFFFFFFFu, pot, 0);
                    for (int l = 1; l < L; ++l) {
                        const double v = __shfl_sync(0xFFFFFFFFu, pot, l);
                        if (v < low) { low = v; best = l; }
                    }
                }
            }
        }
        if (rank == 0 && tid == kStartThreads - 1) p.chosen[q.cplane + c] = sm.draw[par][best].pick;
        if (c + 1 == q.k) break;
        // ---- 3. the winner's distances, a warp per block of the sums, eight lanes per point; the block's sum to all ----
        for (int blk = warp; blk < mb; blk += kStartWarps) {
            double w = sm.raw[b0 + blk];
            if ((sm.touched[blk] >> best) & 1u) {
                const int base = blk * kSumBlock, cnt = min(kSumBlock, n_rows - base), eighth = lane & 7;
                double y[2][8];
#pragma unroll
                for (int h = 0; h < 2; ++h) widen8<kHalf>(sm.trial[near_piece(best, eighth + 8 * h)], y[h]);
                int m = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool marked = (sm.mask[base + e * 32 + lane] >> best) & 1;
                    const unsigned who = __ballot_sync(0xFFFFFFFFu, marked);
                    if (marked) sm.list[warp][m + __popc(who & ((1u << lane) - 1u))] = (uint8_t)(e * 32 + lane);
                    m += __popc(who);
                }
                __syncwarp();
                const int unit = sm.draw[par][best].unit;
                int first_at = kSumBlock;                       // first point that gets a smaller distance
#pragma unroll 2
                for (int j0 = 0; j0 < m; j0 += 4) {
                    const int j = j0 + (lane >> 3), at = sm.list[warp][min(j, m - 1)], i = base + at;
                    double d = sum_parts(start_dist_part<kHalf>(sm.rows, i, eighth, y));
                    bool did = false;
                    if (j < m && eighth == 0) {
                        // Rows that are multiples of 2^u: their distance is one of 2^2u, and so is every partial sum. Below 2^(53 + 2u)
                        // none of them is rounded, and the order of the sum does not matter; else the defining order.
                        const int u = min(unit, (int)sm.unit[i]);
                        const double exact_below = u > -128 ? __hiloint2double((1023 + 52 + 2 * u) << 20, 0) : 0.0;
                        if (!(d < exact_below)) d = start_dist<kHalf>(sm.rows, i, sm.trial, best);
                        if (d < sm.closest[i] || c == 0) {
                            did = true;
                            sm.closest[i] = d;
                            // (a norm that fp32 does not hold: the product decides nothing; nothing is nearer than zero)
                            sm.bar[i] = !(sm.norm[i] <= 1e37f) ? -CUDART_INF_F
                                      : d == 0.0 ? CUDART_INF_F : sm.norm[i] * (1.f - kPairErr) - __double2float_ru(d);
                        }
                    }
                    first_at = min(first_at, did ? at : kSumBlock);
                }
                first_at = __reduce_min_sync(0xFFFFFFFFu, first_at);
                __syncwarp();
                if (first_at < kSumBlock) {
                    if (lane == 0) w = run_sums(sm.closest + base, sm.run + base, first_at, cnt, first_at > 0 ? sm.run[base + first_at - 1] : 0.0);
                    w = __shfl_sync(0xFFFFFFFFu, w, 0);
                }
            }
            if (lane < n_blk) send_double(in_block(shared_addr(&sm.raw[b0 + blk]), lane), in_block(shared_addr(&sm.arrived[kSums]), lane), w);
        }
        // ---- 4. the blocks' running sums; the next trial points, a warp per draw: the block that owns a drawn point sends
        // its row to all ----
        const int l = warp;
        const uint32_t word = km_word(p, (uint32_t)l, kTagStart, q.stream, (uint32_t)(c + 1));
        await(kSums, (uint32_t)par);
        if (tid == 0) run_sums(sm.raw, sm.pre, 0, nb, 0.0);
        __syncthreads();
        if (tid < kStartBlocks) sm.touched[tid] = 0u;
        if (tid >= 32 && tid < 32 + 2 * kStartTrials) sm.own_gain[par][0][tid - 32] = 0.f;      // (for the centre after the next)
        if (l < q.L) {
            const double target = __dmul_rn(((double)word + 0.5) * (1.0 / 4294967296.0), sm.pre[nb - 1]);
            int blk = nb;                                   // first block whose running sum exceeds the target
#pragma unroll
            for (int o = kStartSums - 32; o >= 0; o -= 32) {
                const unsigned over = __ballot_sync(0xFFFFFFFFu, o + lane < nb && sm.pre[min(o + lane, nb - 1)] > target);
                if (over) blk = o + __ffs(over) - 1;
            }
            const bool none = blk == nb;                    // rounding left no point beyond the target: the last one
            if (none) blk = nb - 1;
            if (blk >= b0 && blk < b0 + mb) {
                const int base = (blk - b0) * kSumBlock, cnt = min(kSumBlock, n_rows - base), h = lane & 15;
                const double before = blk > 0 ? sm.pre[blk - 1] : 0.0;
                int at = cnt - 1;                           // first point of the block with offset + running sum beyond it
#pragma unroll
                for (int e = kSumBlock / 32 - 1; e >= 0; --e) {
                    const unsigned over = __ballot_sync(0xFFFFFFFFu, !none && e * 32 + lane < cnt && __dadd_rn(before, sm.run[base + e * 32 + lane]) > target);
                    if (over) at = e * 32 + __ffs(over) - 1;
                }
                const uint4 piece = sm.rows[near_piece(base + at, h)];
                const uint32_t to = shared_addr(&sm.trial[near_piece(l, h)]), bar = shared_addr(&sm.arrived[kDraws]);
#pragma unroll
                for (int b = 0; b < kStartMaxCluster; b += 2)       // half a warp a block
                    if (b + (lane >> 4) < n_blk) send4(in_block(to, b + (lane >> 4)), in_block(bar, b + (lane >> 4)), piece);
                if (lane < n_blk)
                    send4(in_block(shared_addr(&sm.draw[par ^ 1][l]), lane), in_block(bar, lane),
                          make_uint4(__float_as_uint(sm.norm[base + at]), (uint32_t)(row0 + base + at), (uint32_t)(int)sm.unit[base + at], 0u));
            }
        }
        // (read here: in the next centre thread 0 writes these sums again once the messages are there, which wait for the warps that send some
        // and not for the others)
        slack = (float)(1e-11 * sm.pre[nb - 1]);
        await(kDraws, (uint32_t)par);
        if (__syncthreads_or(sm.failed)) break;
    }
    tc_fence_before();
    cluster_barrier();                                      // (a block's shared memory stays while another may send to it)
    tc_fence_after();
    if (sm.failed)                                          // messages that were not waited for: they take a microsecond
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(kTmemCols));
    if (tid == 0 && sm.failed) p.chosen[q.cplane] = -1;
}

// How many blocks share a pair's sample in km_start_kernel; 0: the sample does not fit, or the device has no room for
// such a cluster. Sixteen where every pair gets its cluster at once; eight halve the wait of many pairs.
template <bool kHalf>
int start_cluster(const KmeansParams &p, int pairs)
{
    const int nb = (p.n_init_max + kSumBlock - 1) / kSumBlock;
    if (nb > kStartSums || p.trials_max > kStartTrials) return 0;
    const int n_blk = nb <= kStartBlocks * 8 && pairs > 8 ? 8 : kStartMaxCluster;
    const void *fn = (const void *)km_start_kernel<kHalf>;
    static std::atomic<unsigned long long> done;
    if (ensure_dynamic_smem(fn, (int)sizeof(StartSmem), done) != cudaSuccess
        || cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    cudaLaunchAttribute dims;
    dims.id = cudaLaunchAttributeClusterDimension;
    dims.val.clusterDim.x = n_blk;
    dims.val.clusterDim.y = dims.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pairs * n_blk);
    cfg.blockDim = dim3(kStartThreads);
    cfg.dynamicSmemBytes = sizeof(StartSmem);
    cfg.attrs = &dims;
    cfg.numAttrs = 1;
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, km_start_kernel<kHalf>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return fit > 0 ? n_blk : 0;
}

template <bool kHalf>
cudaError_t launch_start(const KmeansParams &p, int pairs, int n_blk, cudaStream_t s)
{
    cudaLaunchAttribute dims;
    dims.id = cudaLaunchAttributeClusterDimension;
    dims.val.clusterDim.x = n_blk;
    dims.val.clusterDim.y = dims.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pairs * n_blk);
    cfg.blockDim = dim3(kStartThreads);
    cfg.dynamicSmemBytes = sizeof(StartSmem);
    cfg.stream = s;
    cfg.attrs = &dims;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, km_start_kernel<kHalf>, p);
}

// ---- 3. minibatch steps ----
// A step is five kernels: the scan for the nearest centres (nearest.cuh), the fp64 distance to the one found,
// the minibatch ordered by centre, the update, the reassignment of starved centres. The inertia of a
// minibatch is a sum of `batch` terms in order -- 4096 dependent additions, 18 us -- and only decides whether
// the next step's update is still made. An extra block per pair in four of the kernels from the update on takes
// a part of it, so it is over when the next update starts and costs no time of its own; from then on a fit
// that has stopped does nothing. At 4 pairs, batch 4096 and 2048 centres a step was 0.94 ms (0.84 of it fp64
// distances to every centre).
__device__ __forceinline__ bool pair_active(const KmeansParams &p, const Pair &q, int t)
{
    return t < q.t_max && !p.state[q.id].stopped;
}

// Four components of a centre per lane of a warp: the fp64 centre, its 16-bit rounding and its bound constants.
template <bool kHalf>
__device__ __forceinline__ void store_centre(const KmeansParams &p, size_t centre, const double (&v)[4])
{
    const int lane = threadIdx.x & 31;
    uint16_t hi[4];
    float n = 0.f, m = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        hi[e] = double_to_elem<kHalf>(v[e]);
        const float r = (float)(v[e] - elem_to_double<kHalf>(hi[e]));
        n = fmaf((float)v[e], (float)v[e], n);
        m = fmaf(r, r, m);
    }
    n = warp_sum(n);
    m = 1.00001f * sqrtf(warp_sum(m));
    const float bias = centre_bias<kHalf>(n);
    const bool fits = bias > -kNearFar;
    double2 *to = reinterpret_cast<double2 *>(p.centres64 + centre * kHeadDim + 4 * lane);
    to[0] = make_double2(v[0], v[1]);
    to[1] = make_double2(v[2], v[3]);
    reinterpret_cast<uint2 *>(p.centre_hi + centre * kHeadDim)[lane] =
        fits ? make_uint2((uint32_t)hi[0] | ((uint32_t)hi[1] << 16), (uint32_t)hi[2] | ((uint32_t)hi[3] << 16)) : make_uint2(0u, 0u);
    if (lane == 0) p.centre_bias[centre] = make_float2(bias, fits ? m : 0.f);
}

// The centres that the start chose (sample indices), their counts and the fits' state at zero. A warp per centre.
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
km_prepare_kernel(KmeansParams p)
{
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    const int u = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool lost = p.chosen[q.cplane] < 0;               // the start gave up on a message (never expected): no centres, no steps
    if (blockIdx.x == 0 && threadIdx.x == 0) p.state[q.id] = KmeansState{0.0, 0.0, 0.0, 0, lost ? -1 : 0, lost ? 1 : 0, 0};
    if (u >= q.k) return;
    const int row = p.perm[q.plane + (lost ? 0 : p.chosen[q.cplane + u])];
    const uint2 w = reinterpret_cast<const uint2 *>(p.k_prompt + (q.plane + row) * kHeadDim)[lane];
    double v[4] = {(double)elem_lo<kHalf>(w.x), (double)elem_hi<kHalf>(w.x), (double)elem_lo<kHalf>(w.y), (double)elem_hi<kHalf>(w.y)};
    if (lost) v[0] = v[1] = v[2] = v[3] = CUDART_NAN;
    store_centre<kHalf>(p, q.cplane + u, v);
    if (lane == 0) p.count[q.cplane + u] = 0.0;
}

// Parts [part, part_end) of kInertiaParts of the inertia of step t, one block per pair; after the last part the averaged
// inertia and the stopping rule. A part's terms go through shared memory: one thread adds them in order.
// The parts ride on the update, the reassignment, the next step's resolve and its sorting kernel, in sixteenths of the minibatch
// by what these kernels take without them (16, 5, 13, 13 us; a sixteenth takes 1.2). None rides on the scan, whose blocks
// fill the device: a fifth of the terms there made 300 blocks for 296 places (40 us, now 35).
constexpr int kInertiaParts = 4, kInertiaTerms = 4096 * 6 / 16 + 1;
__device__ __forceinline__ int inertia_cut(int part, int batch)
{
    const int sixteenths = part <= 0 ? 0 : part == 1 ? 6 : part == 2 ? 7 : part == 3 ? 12 : 16;
    return (int)((long long)sixteenths * batch / 16);
}
__device__ __forceinline__ void km_inertia(const KmeansParams &p, const Pair &q, int t, int part, int part_end, double *term_s)
{
    if (t < 0 || !pair_active(p, q, t)) return;
    KmeansState &st = p.state[q.id];
    const double *dist = p.dist + ((size_t)(t & 1) * p.n_seqs * p.n_kv + q.id) * p.batch;
    double sum = part > 0 ? st.partial : 0.0;
    for (; part < part_end; ++part) {
        const int lo = inertia_cut(part, p.batch), n = inertia_cut(part + 1, p.batch) - lo;
        __syncthreads();
        for (int s = threadIdx.x; s < n; s += blockDim.x) term_s[s] = dist[lo + s];
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll 16
            for (int s = 0; s < n; ++s) sum = __dadd_rn(sum, term_s[s]);
        }
    }
    if (threadIdx.x != 0) return;
    st.partial = sum;
    if (part < kInertiaParts) return;
    double alpha = __ddiv_rn(__dmul_rn(2.0, (double)p.batch), __dadd_rn((double)q.N, 1.0));
    if (alpha > 1.0) alpha = 1.0;
    const double per_point = __ddiv_rn(sum, (double)p.batch);
    const double ewa = t == 0 ? per_point
                              : __dadd_rn(__dmul_rn(st.ewa, __dsub_rn(1.0, alpha)), __dmul_rn(per_point, alpha));
    st.ewa = ewa;
    st.steps += 1;
    if (t == 0 || ewa < st.ewa_min) { st.ewa_min = ewa; st.bad = 0; }
    else if (++st.bad >= p.patience) st.stopped = 1;
}

// After the last step: what is left of its inertia (its update and reassignment kernels took two parts).
__global__ void __launch_bounds__(kThreads)
km_last_inertia_kernel(KmeansParams p, int t)
{
    __shared__ double term_s[kInertiaTerms];
    step_wait();
    km_inertia(p, pair_of(p, blockIdx.x / p.n_kv, blockIdx.x % p.n_kv), t, 2, kInertiaParts, term_s);
}

// A pair's minibatch as tiles of 128 points, its centres as tiles of 128: their products in row-major order are cut
// into equal ranges, one per block of the pair. A block leaves one NearTop per point and tile of points it touches.
struct ScanSplit {
    int k_tiles, units, blocks;
    __device__ int start(int i) const { return (int)((long long)i * units / blocks); }
    __device__ int block_of(int unit) const { return (int)(((long long)(unit + 1) * blocks - 1) / units); }
};
__device__ __forceinline__ ScanSplit scan_split(const KmeansParams &p, const Pair &q)
{
    ScanSplit s;
    s.k_tiles = (q.k + kNearTile - 1) / kNearTile;
    s.units = s.k_tiles * ((p.batch + kNearPoints - 1) / kNearPoints);
    s.blocks = min(p.scan_blocks, s.units);
    return s;
}

// Draw the minibatch and scan the centres for each point's nearest.
template <bool kHalf>
__global__ void __launch_bounds__(kNearThreads, 2)
km_scan_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(1024) unsigned char near_smem[];
    NearSmem &sm = *reinterpret_cast<NearSmem *>(near_smem);
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    const int tid = threadIdx.x;
    if (!pair_active(p, q, t)) return;
    const ScanSplit sp = scan_split(p, q);
    if ((int)blockIdx.x >= sp.blocks) return;
    const uint16_t *keys = p.k_prompt + q.plane * kHeadDim;
    const uint4 *hi = reinterpret_cast<const uint4 *>(p.centre_hi + q.cplane * kHeadDim);
    const float2 *bias = p.centre_bias + q.cplane;
    const int end = sp.start(blockIdx.x + 1);
    uint32_t uses[2] = {0u, 0u};
    near_open_block(sm);
    for (int unit = sp.start(blockIdx.x); unit < end;) {
        const int tile = unit / sp.k_tiles, k0 = unit - tile * sp.k_tiles, k1 = min(sp.k_tiles, k0 + end - unit);
        const int s = tile * kNearPoints + tid;
        if (tid < kNearPoints) {
            sm.idx[tid] = km_index(km_word(p, (uint32_t)(s < p.batch ? s : 0), kTagBatch, q.stream, (uint32_t)t), q.N);
            if (k0 == 0 && s < p.batch) p.idx[(size_t)q.id * p.batch + s] = sm.idx[tid];
        }
        __syncthreads();
        near_scan<kHalf>(sm, [&](int i) { return keys + (size_t)sm.idx[i] * kHeadDim; }, k0 * kNearTile, min(k1 * kNearTile, q.k), uses,
                         [&](int stage, int slot, int base, int n) {
#pragma unroll
                             for (int m = 0; m < kNearTile * 16 / kNearThreads; ++m) {
                                 const int e = m * kNearThreads + tid, row = e >> 4;
                                 copy16_or_zero(shared_addr(sm.centres[stage] + near_byte(row, e & 15)), hi + (size_t)(base + min(row, n - 1)) * 16 + (e & 15), row < n);
                             }
                             if (tid < kNearTile) sm.bias[slot][tid] = tid < n ? bias[base + tid] : make_float2(kNearFar, 0.f);
                         });
        if (tid < kNearPoints && s < p.batch) {
            const int seg = (int)blockIdx.x - sp.block_of(tile * sp.k_tiles);
            p.near_top[((size_t)q.id * p.scan_segs + seg) * p.batch + s] = sm.top[tid];
            if (k0 == 0) p.near_nx[(size_t)q.id * p.batch + s] = sm.nx[tid];
        }
        unit += k1 - k0;
        __syncthreads();                                    // sm.top, sm.nx and sm.idx are read
    }
    near_close_block(sm);
}

// The nearest centre of each minibatch point and the fp64 distance to it: the scan's results merged, the
// candidates that the bounds leave open compared in fp64. A block takes 64 points, eight per warp: the terms of each distance
// are formed by all lanes (coalesced reads, four conversions a lane), then a thread per point adds them up in order. Bound by the
// latency of scattered reads: with 32 points per warp, one after another, 5 % of the warps were resident (4 x 4096 points: 21 us,
// now 13).
constexpr int kResolveThreads = 256, kResolveWarps = kResolveThreads / 32, kResolvePoints = 64, kTermPitch = kHeadDim + 1;
// Points of a block up to which they go through all centres one by one: eight warps at about 37 us a point and 512 centres, against 200
// for all of the block's together.
constexpr int kResolveFewOpen = 24;
struct ResolveSmem {
    double term[kResolvePoints][kTermPitch];
    __align__(16) double tmp[kResolveWarps][kHeadDim];
    double dist[2 * kResolvePoints];                        // of the listed candidates, or of the open points
    int2 list[2 * kResolvePoints];                          // (point, centre)
    int found[kResolvePoints];                              // nearest centres of the open points
    int point[kResolvePoints], centre[kResolvePoints];
    int n_list, n_open;
};
// Squared differences of a row (16-bit values) and a centre in each dimension, by a warp.
template <bool kHalf>
__device__ __forceinline__ void resolve_terms(const uint16_t *x, const double *c, double *term)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const double d = __dsub_rn(elem_to_double<kHalf>(__ldg(x + 32 * e + lane)), c[32 * e + lane]);
        term[32 * e + lane] = __dmul_rn(d, d);
    }
}
template <bool kHalf>
__global__ void __launch_bounds__(kResolveThreads)
km_resolve_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ResolveSmem &sm = *reinterpret_cast<ResolveSmem *>(smem_raw);
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    if (blockIdx.x == gridDim.x - 1) {
        km_inertia(p, q, t - 1, 2, 3, &sm.term[0][0]);
        return;
    }
    if (!pair_active(p, q, t)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, s = blockIdx.x * kResolvePoints + tid;
    const bool live = tid < kResolvePoints && s < p.batch;
    const size_t at = (size_t)q.id * p.batch + (live ? s : 0);
    const double *cen = p.centres64 + q.cplane * kHeadDim;
    const uint16_t *keys = p.k_prompt + q.plane * kHeadDim;
    if (tid == 0) sm.n_list = sm.n_open = 0;
    __syncthreads();
    const int point = p.idx[at];
    int arg = 0, second = -1, third = -1, open_at = -1;     // places in the lists
    NearTop top = near_none(0);
    if (tid < kResolvePoints) {
        const ScanSplit sp = scan_split(p, q);
        const int tile = (live ? s : 0) / kNearPoints;
        const int segs = sp.block_of(tile * sp.k_tiles + sp.k_tiles - 1) - sp.block_of(tile * sp.k_tiles) + 1;
        for (int seg = 0; seg < segs; ++seg) near_merge(top, p.near_top[((size_t)q.id * p.scan_segs + seg) * p.batch + (live ? s : 0)]);
        arg = top.i1;
        sm.point[tid] = point;
        sm.centre[tid] = arg;
        if (live) {
            if (near_open(top, p.near_nx[at])) {
                open_at = atomicAdd(&sm.n_open, 1);
            } else {
                if (!(top.t2 > top.upper)) sm.list[second = atomicAdd(&sm.n_list, 1)] = make_int2(point, top.i2);
                if (!(top.t3 > top.upper)) sm.list[third = atomicAdd(&sm.n_list, 1)] = make_int2(point, top.i3);
            }
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int l = 0; l < kResolvePoints / kResolveWarps; ++l) {
        const int i = warp * (kResolvePoints / kResolveWarps) + l;
        resolve_terms<kHalf>(keys + (size_t)sm.point[i] * kHeadDim, cen + (size_t)sm.centre[i] * kHeadDim, sm.term[i]);
    }
    const int n_list = sm.n_list, n_open = sm.n_open;
    for (int e = warp; e < n_list; e += kResolveWarps) {    // second and third candidates, a warp each
        resolve_terms<kHalf>(keys + (size_t)sm.list[e].x * kHeadDim, cen + (size_t)sm.list[e].y * kHeadDim, sm.tmp[warp]);
        __syncwarp();
        if (lane == 0) {
            double d = 0.0;
#pragma unroll 16
            for (int u = 0; u < kHeadDim; ++u) d = __dadd_rn(d, sm.tmp[warp][u]);
            sm.dist[e] = d;
        }
        __syncwarp();
    }
    __syncthreads();
    double best = 0.0;
    if (tid < kResolvePoints) {
#pragma unroll 16
        for (int d = 0; d < kHeadDim; ++d) best = __dadd_rn(best, sm.term[tid][d]);
        if (second >= 0) {
            const double d2 = sm.dist[second];
            if (d2 < best || (d2 == best && top.i2 < arg)) { best = d2; arg = top.i2; }
        }
        if (third >= 0) {
            const double d3 = sm.dist[third];
            if (d3 < best || (d3 == best && top.i3 < arg)) { best = d3; arg = top.i3; }
        }
    }
    if (n_open > kResolveFewOpen) {
        double d;
        const int u = near_scan_tiles<kHalf, kResolveThreads, 1>(reinterpret_cast<const uint4 *>(keys + (size_t)point * kHeadDim), open_at >= 0, cen, q.k,
                                                                 reinterpret_cast<double (*)[kHeadDim]>(smem_raw), d);
        if (open_at >= 0) { best = d; arg = u; }
    } else if (n_open > 0) {
        __syncthreads();                                    // the terms and the candidates' distances have been read
        if (open_at >= 0) sm.point[open_at] = point;
        __syncthreads();
        for (int e = warp; e < n_open; e += kResolveWarps) {
            double d;
            const int u = near_scan_exact<kHalf>(reinterpret_cast<const uint4 *>(keys + (size_t)sm.point[e] * kHeadDim), cen, q.k, sm.tmp[warp], d);
            if (lane == 0) { sm.dist[e] = d; sm.found[e] = u; }
        }
        __syncthreads();
        if (open_at >= 0) { best = sm.dist[open_at]; arg = sm.found[open_at]; }
    }
    if (live) {
        p.label[at] = arg;
        p.dist[((size_t)(t & 1) * p.n_seqs * p.n_kv + q.id) * p.batch + s] = best;
    }
}

// The minibatch ordered by (label, slot), one block per pair: two stable counting passes over the label's digits
// (8 bits each: a fit has at most 28544 centres), then where each label starts. A thread holds four entries; ranks of
// equal digits come from the warp (in order) and from counts of the warps before. (A bitonic sort of the same keys
// took 24 us.)
constexpr int kSortThreads = 1024, kSortKeys = 4096, kSortBits = 8, kSortDigits = 1 << kSortBits, kSortWarps = kSortThreads / 32;
struct SortSmem {
    uint32_t key[2][kSortKeys];                             // label << 12 | slot
    uint16_t count[kSortDigits][kSortWarps + 2];
    int scan[33];
};
__global__ void __launch_bounds__(kSortThreads)
km_sort_batch_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SortSmem &sm = *reinterpret_cast<SortSmem *>(smem_raw);
    step_wait();
    const int pairs = p.n_seqs * p.n_kv, pair = blockIdx.x % pairs;
    const Pair q = pair_of(p, pair / p.n_kv, pair % p.n_kv);
    if ((int)blockIdx.x >= pairs) {
        km_inertia(p, q, t - 1, 3, 4, reinterpret_cast<double *>(smem_raw));
        return;
    }
    // one look at the flag for the block: beside it the block above may be stopping this very fit
    if (!__syncthreads_or(threadIdx.x == 0 && pair_active(p, q, t))) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t *idx = p.idx + (size_t)q.id * p.batch;
    uint32_t key[4];                                        // the warp's 128 entries, 32 at a time in order
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int s = warp * 128 + c * 32 + lane;
        key[c] = s < p.batch ? ((uint32_t)p.label[(size_t)q.id * p.batch + s] << 12) | (uint32_t)s : 0xFFFFFFFFu;
    }
    for (int pass = 0; pass < 2; ++pass) {
        const int shift = 12 + pass * kSortBits;
        for (int e = tid; e < kSortDigits * (kSortWarps + 2) / 2; e += kSortThreads) reinterpret_cast<uint32_t *>(&sm.count[0][0])[e] = 0u;
        __syncthreads();
        int digit[4], rank[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (pass == 1) key[c] = sm.key[1][warp * 128 + c * 32 + lane];
            digit[c] = (int)((key[c] >> shift) & (kSortDigits - 1));
            unsigned same = 0xFFFFFFFFu;                    // lanes with the same digit
#pragma unroll
            for (int bit = 0; bit < kSortBits; ++bit) {
                const bool on = (digit[c] >> bit) & 1;
                const unsigned with = __ballot_sync(0xFFFFFFFFu, on);
                same &= on ? with : ~with;
            }
            const unsigned before = same & ((1u << lane) - 1u);
            const int base = sm.count[digit[c]][warp];
            rank[c] = base + __popc(before);
            __syncwarp();
            if (before == 0u) sm.count[digit[c]][warp] = (uint16_t)(base + __popc(same));
            __syncwarp();
        }
        __syncthreads();
        // exclusive prefix over (digit, warp): thread = digit * 4 + part of eight warps
        {
            const int d = tid >> 2, w0 = (tid & 3) * 8;
            int n[8], sum = 0, total;
#pragma unroll
            for (int w = 0; w < 8; ++w) { n[w] = sm.count[d][w0 + w]; sum += n[w]; }
            int at = block_exclusive_scan(sum, sm.scan, total);
#pragma unroll
            for (int w = 0; w < 8; ++w) { sm.count[d][w0 + w] = (uint16_t)at; at += n[w]; }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c) sm.key[pass ^ 1][sm.count[digit[c]][warp] + rank[c]] = key[c];
        __syncthreads();
    }
    int32_t *start = p.start + (size_t)q.id * (p.k_max + 1);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int s = c * kSortThreads + tid;
        const uint32_t mine = sm.key[0][s];
        const int label = min((int)(mine >> 12), q.k);      // (the padding sorts behind every label)
        const int prev = s > 0 ? min((int)(sm.key[0][s - 1] >> 12), q.k) : -1;
        for (int u = prev + 1; u <= label; ++u) start[u] = s;
        if (s == kSortKeys - 1)
            for (int u = label + 1; u <= q.k; ++u) start[u] = kSortKeys;
        if (s < p.batch) p.sorted[(size_t)q.id * kSortKeys + s] = idx[mine & 4095u];
    }
}

// Cumulative-count update, a warp per centre (four dimensions per lane): the centre's new points are added in
// minibatch order; c <- (c * count + sum) / (count + n). The next kAhead rows are on their way while kAhead are added:
// 16 for centres of many points; 4 where a centre has less than eight on average, since 16 take the registers of
// three of four warps (2048 centres of two points were three and a half waves of blocks; 18.5 us, now 16.4).
template <bool kHalf, int kAhead>
__global__ void __launch_bounds__(128, kAhead > 4 ? 4 : 8)
km_batch_update_kernel(KmeansParams p, int t)
{
    __shared__ double term_s[kInertiaTerms];
    step_wait();
    const Pair q = pair_of(p, blockIdx.y / p.n_kv, blockIdx.y % p.n_kv);
    if (blockIdx.x == gridDim.x - 1) {
        km_inertia(p, q, t, 0, 1, term_s);
        return;
    }
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
    int id = point[min(lo + lane, hi - 1)];                 // tokens of the 32 points from `lo` on
    uint2 next[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
        const int tok = __shfl_sync(0xFFFFFFFFu, id, i);
        if (lo + i < hi) next[i] = __ldg(keys + (size_t)tok * 32);
    }
    for (int i0 = lo; i0 < hi; i0 += kAhead) {
        uint2 w[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) w[i] = next[i];
        const int place = (i0 - lo + kAhead) & 31;          // place of the next ones among the 32 of `id`
        if (place == 0) id = point[min(i0 + kAhead + lane, hi - 1)];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const int tok = __shfl_sync(0xFFFFFFFFu, id, place + i);
            if (i0 + kAhead + i < hi) next[i] = __ldg(keys + (size_t)tok * 32);
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
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

// Reassignment of starved centres, one block per pair (and one that takes a part of the inertia).
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
km_reassign_kernel(KmeansParams p, int t)
{
    extern __shared__ __align__(16) int32_t slots[];        // slots[batch], then move_centre[batch / 2]
    __shared__ int scan_s[33];
    __shared__ double cmin_s[kThreads / 32], cmax_s[kThreads / 32];
    step_wait();
    const Pair q = pair_of(p, blockIdx.x, blockIdx.y);
    if (blockIdx.z == 1) {
        km_inertia(p, q, t, 1, 2, reinterpret_cast<double *>(slots));
        return;
    }
    if (!(p.ratio > 0.0) || !pair_active(p, q, t)) return;
    const int tid = threadIdx.x;
    int32_t *move_centre = slots + p.batch;
    double *count = p.count + q.cplane;
    auto reduce = [&](double v, bool smallest, double *scratch) {     // any order gives the same
        for (int o = 16; o > 0; o >>= 1) {
            const double w = __shfl_xor_sync(0xffffffffu, v, o);
            if (smallest ? w < v : w > v) v = w;
        }
        __syncthreads();
        if ((tid & 31) == 0) scratch[tid >> 5] = v;
        __syncthreads();
        for (int w = 0; w < kThreads / 32; ++w)
            if (smallest ? scratch[w] < v : scratch[w] > v) v = scratch[w];
        return v;
    };
    double cmin = INFINITY, cmax = 0.0;
    for (int u = tid; u < q.k; u += kThreads) {
        const double v = count[u];
        if (v < cmin) cmin = v;
        if (v > cmax) cmax = v;
    }
    cmin = reduce(cmin, true, cmin_s);
    const long long period = 10 + (long long)floor(cmin);
    if (((long long)t + 1) % period != 0) return;
    cmax = reduce(cmax, false, cmax_s);
    // the starved centres in order, at most batch / 2 of them; the smallest count among the others
    const double thr = __dmul_rn(p.ratio, cmax);
    const int cap = p.batch / 2;
    int n_move = 0;
    double keep_min = INFINITY;
    for (int u0 = 0; u0 < q.k; u0 += kThreads) {
        const int u = u0 + tid;
        const double v = u < q.k ? count[u] : INFINITY;
        const bool starved = u < q.k && v < thr;
        int total;
        const int at = n_move + block_exclusive_scan(starved ? 1 : 0, scan_s, total);
        if (starved && at < cap) move_centre[at] = u;
        else if (u < q.k && v < keep_min) keep_min = v;
        n_move += total;
    }
    n_move = min(n_move, cap);
    if (n_move == 0) return;
    keep_min = reduce(keep_min, true, cmin_s);
    for (int s = tid; s < p.batch; s += kThreads) slots[s] = s;
    __syncthreads();
    if (tid == 0)
        for (int i = 0; i < n_move; ++i) {
            const int r = i + km_index(km_word(p, (uint32_t)i, kTagMove, q.stream, (uint32_t)t), p.batch - i);
            const int tmp = slots[i];
            slots[i] = slots[r];
            slots[r] = tmp;
        }
    __syncthreads();
    for (int i = tid; i < n_move; i += kThreads) count[move_centre[i]] = keep_min;
    const int32_t *idx = p.idx + (size_t)q.id * p.batch;
    for (int i = tid >> 5; i < n_move; i += kThreads / 32) {     // the moved centres jump onto minibatch points
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
    const int n_blk = start_cluster<kHalf>(p, pairs);
    if (n_blk > 0) {
        if ((err = launch_start<kHalf>(p, pairs, n_blk, s)) != cudaSuccess) return err;
    } else {
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
    }
    const dim3 threads(kThreads);
    if ((err = launch_step(km_prepare_kernel<kHalf>, dim3((p.k_max + kThreads / 32 - 1) / (kThreads / 32), pairs), threads, 0, s, p)) != cudaSuccess) return err;
    static std::atomic<unsigned long long> scan_done, resolve_done, sort_done;
    if ((err = ensure_dynamic_smem((const void *)km_scan_kernel<kHalf>, (int)sizeof(NearSmem), scan_done)) != cudaSuccess) return err;
    if ((err = ensure_dynamic_smem((const void *)km_resolve_kernel<kHalf>, (int)sizeof(ResolveSmem), resolve_done)) != cudaSuccess) return err;
    if ((err = ensure_dynamic_smem((const void *)km_sort_batch_kernel, (int)sizeof(SortSmem), sort_done)) != cudaSuccess) return err;
    const size_t move_smem = std::max(sizeof(int32_t) * ((size_t)p.batch + (size_t)p.batch / 2 + 1), sizeof(double) * (size_t)kInertiaTerms);
    const dim3 resolve_grid((p.batch + kResolvePoints - 1) / kResolvePoints + 1, pairs);
    int t = 0;
    for (; t < p.t_max_max; ++t) {
        if ((err = launch_step(km_scan_kernel<kHalf>, dim3(p.scan_blocks, pairs), dim3(kNearThreads), sizeof(NearSmem), s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_resolve_kernel<kHalf>, resolve_grid, dim3(kResolveThreads), sizeof(ResolveSmem), s, p, t)) != cudaSuccess) return err;
        if ((err = launch_step(km_sort_batch_kernel, dim3(2 * pairs), dim3(kSortThreads), sizeof(SortSmem), s, p, t)) != cudaSuccess) return err;
        const dim3 update_grid((p.k_max + 3) / 4 + 1, pairs);
        err = p.batch < 8 * p.k_max ? launch_step(km_batch_update_kernel<kHalf, 4>, update_grid, dim3(128), 0, s, p, t)
                                    : launch_step(km_batch_update_kernel<kHalf, 16>, update_grid, dim3(128), 0, s, p, t);
        if (err != cudaSuccess) return err;
        if ((err = launch_step(km_reassign_kernel<kHalf>, dim3(B, H, 2), threads, move_smem, s, p, t)) != cudaSuccess) return err;
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
    if ((err = launch_step(km_last_inertia_kernel, dim3(pairs), threads, 0, s, p, t - 1)) != cudaSuccess) return err;   // counts the last step
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
