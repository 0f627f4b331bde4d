// santapp_build_teams: contiguous parents (Algorithm 4) and actual-key teams (Algorithm 2),
// written as a team-contiguous copy of K/V with CSR offsets. Preparation path, run once after
// prefill. The teams are those of fp64 distances evaluated in a fixed order (select_rows.cuh says how
// they are found without evaluating most of them).
//
// One kernel does all of it (parent_teams.cuh): a parent's rows keep their range of the packed order, so a
// block that knows its parent's owners also knows the parent's row offsets, and nothing has to be scanned
// over the sequence or read a second time: K goes through shared memory once, V is copied from its old
// place to its new one. 32K keys, 4 KV heads, P = 512, R = 32: 641 us in three kernels with fp64 distances, now 91.
#include <algorithm>

#include "parent_teams.cuh"

namespace santapp {

namespace {

__device__ __forceinline__ bool contiguous_parent(const BuildParams &p, int parent, int b, int j, ParentRows &t)
{
    const int64_t row0 = p.bv.seq_row_off[b];
    const int N = (int)(p.bv.seq_row_off[b + 1] - row0);
    t.s0 = parent * p.parent_size;
    if (t.s0 >= N) return false;
    t.nC = min(p.parent_size, N - t.s0);
    t.r = min(p.reps, t.nC);
    t.k_prompt = p.k_prompt;
    t.v_prompt = p.v_prompt;
    t.k_packed = p.k_packed;
    t.v_packed = p.v_packed;
    t.rep_keys = p.rep_keys;
    t.row_token = p.row_token;
    t.plane = (size_t)j * p.bv.rows_total + row0;
    t.members = nullptr;
    const int64_t team0 = p.bv.seq_team_off[b];
    const int team_local0 = parent * p.teams_per_full_parent;
    t.csr = p.team_row_start + (size_t)j * (p.bv.teams_total + p.bv.n_seqs) + team0 + b + team_local0;
    t.rep0 = (size_t)j * p.bv.teams_total + team0 + team_local0;
    t.abs_max = p.rep_abs_max + (size_t)j * p.bv.n_seqs + b;
    return true;
}

__device__ __forceinline__ void first_parent_writes(const BuildParams &p, int b, int j, const ParentRows &t)
{
    t.csr[0] = 0;
    if (p.team_count) p.team_count[(size_t)j * p.bv.n_seqs + b] = (int)(p.bv.seq_team_off[b + 1] - p.bv.seq_team_off[b]);
}

__host__ __device__ constexpr int small_warps(int rows) { return rows <= 16 ? 4 : 2; }
template <int kRows, bool kHalf>
__global__ void __launch_bounds__(small_warps(kRows) * 32)
build_small_kernel(BuildParams p)
{
    constexpr int kSmallWarps = small_warps(kRows);
    __shared__ SmallSmem<kRows> sm[kSmallWarps];
    step_wait();
    const int warp = threadIdx.x >> 5, parent = blockIdx.x * kSmallWarps + warp, b = blockIdx.y, j = blockIdx.z;
    ParentRows t;
    if (!contiguous_parent(p, parent, b, j, t)) return;
    small_parent<kRows, kHalf>(t, sm[warp]);
    if (parent == 0 && threadIdx.x == 0) first_parent_writes(p, b, j, t);
}

template <int kWarps, int kRpt, bool kHalf>
__global__ void __launch_bounds__(32 * kWarps, large_blocks(kWarps, kRpt))
build_large_kernel(BuildParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    step_wait();
    const int parent = blockIdx.x, b = blockIdx.y, j = blockIdx.z;
    ParentRows t;
    if (!contiguous_parent(p, parent, b, j, t)) return;
    large_parent<kWarps, kRpt, kHalf>(t, *reinterpret_cast<LargeSmem<kWarps, kRpt> *>(smem_raw));
    if (parent == 0 && threadIdx.x == 0) first_parent_writes(p, b, j, t);
}

// Centroid-guided baseline of the paper's routing diagnostic, on the contiguous parents of
// Algorithm 4: one group per parent, routed by the arithmetic mean of its keys. A block per
// (parent, sequence, KV head), a thread per dimension: the mean is the fp64 sum in token order
// divided by the count, stored like every routing key as a 16-bit element (fp64 -> fp32 to nearest,
// then fp32 -> bf16 or fp16 to nearest even). Rows keep their token order, so the packed copies are copies.
template <bool kHalf>
__global__ void __launch_bounds__(kHeadDim)
group_mean_kernel(BuildParams p)
{
    const int parent = blockIdx.x, b = blockIdx.y, j = blockIdx.z, d = threadIdx.x;
    const int64_t row0 = p.bv.seq_row_off[b];
    const int N = (int)(p.bv.seq_row_off[b + 1] - row0);
    const int n_parents = (N + p.parent_size - 1) / p.parent_size;
    if (parent >= n_parents) return;
    const int lo = parent * p.parent_size, hi = min(lo + p.parent_size, N);
    const size_t plane = (size_t)j * p.bv.rows_total + (size_t)row0;
    const uint16_t *k = p.k_prompt + plane * kHeadDim;
    double sum = 0.0;
    for (int i = lo; i < hi; ++i) sum = __dadd_rn(sum, elem_to_double<kHalf>(k[(size_t)i * kHeadDim + d]));
    const int64_t team0 = p.bv.seq_team_off[b];                     // one team per parent
    p.rep_keys[((size_t)j * p.bv.teams_total + (size_t)team0 + parent) * kHeadDim + d] =
        double_to_elem<kHalf>(__ddiv_rn(sum, (double)(hi - lo)));
    int32_t *csr = p.team_row_start + (size_t)j * (p.bv.teams_total + p.bv.n_seqs) + team0 + b;
    if (d == 0) {
        csr[parent] = lo;
        if (parent == n_parents - 1) csr[n_parents] = N;
        if (parent == 0 && p.team_count) p.team_count[(size_t)j * p.bv.n_seqs + b] = n_parents;
    }
    for (int i = lo + d; i < hi; i += kHeadDim) p.row_token[plane + i] = i;
    const uint4 *ks = reinterpret_cast<const uint4 *>(p.k_prompt + (plane + lo) * kHeadDim);
    const uint4 *vs = reinterpret_cast<const uint4 *>(p.v_prompt + (plane + lo) * kHeadDim);
    uint4 *kd = reinterpret_cast<uint4 *>(p.k_packed + (plane + lo) * kHeadDim);
    uint4 *vd = reinterpret_cast<uint4 *>(p.v_packed + (plane + lo) * kHeadDim);
    for (int idx = d; idx < (hi - lo) * (kHeadDim / 8); idx += kHeadDim) {
        kd[idx] = ks[idx];
        vd[idx] = vs[idx];
    }
}

template <int kRows, bool kHalf>
cudaError_t launch_small(const BuildParams &p, cudaStream_t s)
{
    constexpr int kSmallWarps = small_warps(kRows);
    const dim3 grid((p.max_parents_per_seq + kSmallWarps - 1) / kSmallWarps, p.bv.n_seqs, p.bv.n_kv);
    return launch_step(build_small_kernel<kRows, kHalf>, grid, dim3(kSmallWarps * 32), 0, s, p);
}
template <int kWarps, int kRpt, bool kHalf>
cudaError_t launch_large(const BuildParams &p, cudaStream_t s)
{
    static std::atomic<unsigned long long> done;
    const int smem = (int)sizeof(LargeSmem<kWarps, kRpt>);
    const cudaError_t err = ensure_dynamic_smem((const void *)build_large_kernel<kWarps, kRpt, kHalf>, smem, done);
    if (err != cudaSuccess) return err;
    return launch_step(build_large_kernel<kWarps, kRpt, kHalf>, dim3(p.max_parents_per_seq, p.bv.n_seqs, p.bv.n_kv), dim3(32 * kWarps), smem, s, p);
}
// Up to 32 rows all distances of a parent are one small product; above, a block whose threads are its rows.
template <bool kHalf>
cudaError_t launch_by_size(const BuildParams &p, cudaStream_t s)
{
    if (p.parent_size <= 16) return launch_small<16, kHalf>(p, s);
    if (p.parent_size <= 32) return launch_small<32, kHalf>(p, s);
    if (p.parent_size <= 64) return launch_large<2, 1, kHalf>(p, s);
    if (p.parent_size <= 128) return launch_large<4, 1, kHalf>(p, s);
    if (p.parent_size <= 256) return launch_large<8, 1, kHalf>(p, s);
    return launch_large<8, 2, kHalf>(p, s);
}

// Offset tables of a batch, handed to the device inside kernel arguments (a copy from host memory takes
// longer than the launch, and would be read again by every replay of a captured graph), and an array to
// set to zero.
constexpr int kTableChunk = 128;
struct TableChunk {
    int32_t first, n;                                       // entries [first, first + n) of each table
    int64_t v[3][kTableChunk];
};
__global__ void __launch_bounds__(kTableChunk)
tables_kernel(const __grid_constant__ TableChunk c, int64_t *t0, int64_t *t1, int64_t *t2, float *zero, int n_zero)
{
    step_wait();
    const int i = threadIdx.x;
    if (i < c.n) {
        t0[c.first + i] = c.v[0][i];
        t1[c.first + i] = c.v[1][i];
        if (t2) t2[c.first + i] = c.v[2][i];
    }
    for (int e = i; e < n_zero; e += kTableChunk) zero[e] = 0.f;
}

}  // namespace

cudaError_t launch_tables(const int64_t *const (&host)[3], int64_t *const (&dev)[3], int entries, float *zero, int n_zero, cudaStream_t s)
{
    for (int first = 0; first < entries; first += kTableChunk) {
        TableChunk c;
        c.first = first;
        c.n = std::min(kTableChunk, entries - first);
        for (int k = 0; k < 3; ++k)
            for (int i = 0; host[k] && i < c.n; ++i) c.v[k][i] = host[k][first + i];
        const cudaError_t err = launch_step(tables_kernel, dim3(1), dim3(kTableChunk), 0, s, c, dev[0], dev[1], dev[2], zero, first == 0 ? n_zero : 0);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

cudaError_t launch_build_groups_mean(const BuildParams &p, cudaStream_t s)
{
    dim3 grid(p.max_parents_per_seq, p.bv.n_seqs, p.bv.n_kv);
    if (p.bv.elem) group_mean_kernel<true><<<grid, kHeadDim, 0, s>>>(p);
    else           group_mean_kernel<false><<<grid, kHeadDim, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_build_teams(const BuildParams &p, cudaStream_t s)
{
    return p.bv.elem ? launch_by_size<true>(p, s) : launch_by_size<false>(p, s);
}

}  // namespace santapp
