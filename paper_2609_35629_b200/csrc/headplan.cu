// Sampling kernel: one block per (sequence, query head) runs select_head (headplan.cuh).
#include "common.cuh"
#include "headplan.cuh"

namespace santapp {

namespace {

// Few heads: 512 threads each, so that every per-thread loop is short (the kernel is a chain of
// dependent steps, not a throughput problem); more heads: 256 threads and four resident blocks per
// SM, then 128 threads and six or seven.
template <int kHeadThreads, bool kHalf>
__global__ void __launch_bounds__(kHeadThreads, kHeadThreads >= 512 ? 1 : 1024 / kHeadThreads)
headplan_kernel(PlanInputs in)
{
    step_wait();
    __shared__ HeadSmem sm;
    trace_mark(in.trace, 1, 0);
    select_head<kHeadThreads, kHeadThreads >= 512 ? 4 : 2, kHalf>(in, blockIdx.x, sm);
    trace_mark(in.trace, 1, 1);
}

}  // namespace

template <bool kHalf>
static cudaError_t launch_headplan_t(const PlanInputs &in, cudaStream_t s)
{
    const int n_heads = in.bv.n_seqs * in.bv.n_q;
    const int sms = attend_grid_size();
    // up to 2048 scores a head 256 threads are faster than 512 (28 layers of 28 heads, 2048 teams: 675 against 693 us), above
    // they are slower (8192 teams: 715 against 592, 4 x 8192: 37.4 against 32.8)
    if (n_heads <= sms && in.y_stride > 2048) return launch_step(headplan_kernel<512, kHalf>, dim3(n_heads), dim3(512), 0, s, in);
    if (n_heads <= 4 * sms) return launch_step(headplan_kernel<256, kHalf>, dim3(n_heads), dim3(256), 0, s, in);
    // Seven blocks share an SM where that saves a wave of them, else six (the shared memory asked for on top leaves room for six): kernel at
    // 32 / 64 / 96 sequences of 28 heads and 2048 tokens, 896, 1792 and 2688 for 888 places with six: 12.8 -> 9.6, 19.9 -> 17.1 and 26.1 -> 23.3 us,
    // lengths from 500 to 16000 13.4 -> 10.1, 19.9 -> 17.1, 26.3 -> 23.6; where both need as many waves seven are slower by up to a
    // hundredth of the step (48 sequences).
    auto waves = [&](int per_sm) { return (n_heads + per_sm * sms - 1) / (per_sm * sms); };
    const bool seven = waves(7) < waves(6);
    return launch_step(headplan_kernel<128, kHalf>, dim3(n_heads), dim3(128), seven ? 0 : 7168, s, in);
}

cudaError_t launch_headplan(const PlanInputs &in, cudaStream_t s)
{
    return in.bv.elem ? launch_headplan_t<true>(in, s) : launch_headplan_t<false>(in, s);
}

}  // namespace santapp
