// V-trace targets of the Corrector (Section 2.3, Eq. V-trace) and the policy-gradient advantage of
// Eq. A3C-V's first line, from the behaviour log-probs the Actor step emits.
//
// The definition is a double sum per start step s; it telescopes into the backward recursion
//   v_s - V(x_s) = delta_s + g_s c_s (v_{s+1} - V(x_{s+1})),   v_n = V(x_n) = bootstrap,
// run from the last step to the first.  Arrays are time-major [n][B], so the lanes of a warp read
// consecutive floats at every step: the kernel moves 4 (5 with per-step discounts) input and 2 output
// floats per step and trajectory and is bound by HBM (by launch latency at the paper's batch sizes).  The recursion runs in double: its
// arithmetic is free next to the memory traffic, and the results then equal the double-precision
// definition up to the final rounding to float.
#include <math.h>

#include <algorithm>

#include "internal.h"

namespace accerl {

namespace {

constexpr int kCols = 32;   // rollouts of a block, one per lane
constexpr int kSteps = 16;  // time steps of a chunk, one warp each

// Many rollouts: one thread each, from the last step to the first.  The recursion is sequential in t but
// its inputs are not: the loads of kAhead steps are issued together (a rollout is one thread, so nothing
// else hides the memory latency).  Bound by HBM for a million rollouts of one step (12 us for 28 MB) and by
// the chain of exps, some 0.17 us a step, where every SM has a few warps only.
constexpr int kAhead = 8;
__global__ void __launch_bounds__(128)
vtrace_rollout_kernel(const float *__restrict__ logp_smaller, const float *__restrict__ logp_original,
                      const float *__restrict__ rewards, const float *__restrict__ values,
                      const float *__restrict__ bootstrap, const float *__restrict__ discounts, int n, int B,
                      float gamma, float rho_hat, float c_hat, float *__restrict__ vs, float *__restrict__ adv)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    double v_next = (double)bootstrap[b];  // V(x_{t+1})
    double vs_next = v_next;               // v_{t+1}
    double carry = 0.0;                    // v_{t+1} - V(x_{t+1})
    for (int t1 = n - 1; t1 >= 0; t1 -= kAhead) {
        float lo[kAhead], ls[kAhead], rw[kAhead], vv[kAhead], dc[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const long long i = (long long)max(t1 - j, 0) * B + b;
            lo[j] = logp_original[i];
            ls[j] = logp_smaller[i];
            rw[j] = rewards[i];
            vv[j] = values[i];
            dc[j] = discounts ? discounts[i] : gamma;
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int t = t1 - j;
            if (t < 0) break;
            const long long i = (long long)t * B + b;
            const double ratio = exp((double)lo[j] - (double)ls[j]);
            const double rho = fmin(ratio, (double)rho_hat), c = fmin(ratio, (double)c_hat);
            const double g = (double)dc[j], v = (double)vv[j], r = (double)rw[j];
            const double delta = rho * (r + g * v_next - v);
            carry = delta + g * c * carry;
            if (adv) adv[i] = (float)(rho * (r + g * vs_next - v));
            vs_next = v + carry;
            vs[i] = (float)vs_next;
            v_next = v;
        }
    }
}

// Few rollouts.  The recursion is sequential in t, but only two multiply-adds a step of it: the ratios (an exp),
// the temporal differences and the advantages of all steps are independent.  So a block takes 32
// rollouts and, from the last step backwards, 16 steps at a time: warp w loads step w of the chunk
// (whole lines: arrays are time-major) and computes rho, g c and delta, the first warp runs the
// recursion over the chunk out of shared memory, and every warp writes its step's results.  The next
// chunk's loads are issued before the recursion of the current one.  A chunk costs about 1 us while
// every SM has a block, whether its steps are used or not.
__global__ void __launch_bounds__(32 * kSteps)
vtrace_kernel(const float *__restrict__ logp_smaller, const float *__restrict__ logp_original,
              const float *__restrict__ rewards, const float *__restrict__ values,
              const float *__restrict__ bootstrap, const float *__restrict__ discounts, int n, int B,
              float gamma, float rho_hat, float c_hat, float *__restrict__ vs, float *__restrict__ adv)
{
    __shared__ double s_delta[kSteps][kCols], s_gc[kSteps][kCols], s_vs[kSteps + 1][kCols];
    __shared__ float s_v[kSteps][kCols], s_tail[2][kCols];  // V of the chunk; V(x) just behind it, by chunk parity
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.x * kCols + lane;
    const bool col = b < B;
    float lo = 0.f, ls = 0.f, rw = 0.f, vv = 0.f, dc = 0.f;
    auto load = [&](int t) {
        if (t < 0 || !col) return;
        const long long i = (long long)t * B + b;
        lo = __ldg(logp_original + i);
        ls = __ldg(logp_smaller + i);
        rw = __ldg(rewards + i);
        vv = __ldg(values + i);
        dc = discounts ? __ldg(discounts + i) : gamma;
    };
    // warp w owns step t1 - w of the chunk that ends at t1
    load(n - 1 - w);
    if (w == 0) {
        const float v = col ? __ldg(bootstrap + b) : 0.f;
        s_tail[0][lane] = v;
        s_vs[0][lane] = (double)v;  // v_{t+1} behind the chunk
    }
    double carry = 0.0;  // v_{t+1} - V(x_{t+1}), held by the first warp
    int par = 0;
    for (int t1 = n - 1; t1 >= 0; t1 -= kSteps, par ^= 1) {
        const int t = t1 - w;
        s_v[w][lane] = vv;
        __syncthreads();
        const double v_next = w == 0 ? (double)s_tail[par][lane] : (double)s_v[w - 1][lane];
        const double ratio = exp((double)lo - (double)ls);
        const double rho = fmin(ratio, (double)rho_hat), c = fmin(ratio, (double)c_hat);
        const double g = (double)dc, v = (double)vv, r = (double)rw;
        s_delta[w][lane] = rho * (r + g * v_next - v);
        s_gc[w][lane] = g * c;
        if (w == kSteps - 1) s_tail[par ^ 1][lane] = vv;
        load(t - kSteps);  // travels while the recursion runs
        __syncthreads();
        if (w == 0) {
#pragma unroll
            for (int j = 0; j < kSteps; ++j) {  // (steps before the first one compute nothing that is kept)
                carry = s_delta[j][lane] + s_gc[j][lane] * carry;
                s_vs[j + 1][lane] = (double)s_v[j][lane] + carry;
            }
        }
        __syncthreads();
        if (t >= 0 && col) {
            const long long i = (long long)t * B + b;
            vs[i] = (float)s_vs[w + 1][lane];
            if (adv) adv[i] = (float)(rho * (r + g * s_vs[w][lane] - v));
        }
        __syncthreads();
        if (w == kSteps - 1) s_vs[0][lane] = s_vs[kSteps][lane];
    }
}

// Which of the two: the time of one thread per rollout grows with the steps (0.17 us each, 0.21 with an
// array of discounts to load, half as much again where the inputs do not fit L2), that of one warp per step
// with the chunks of 16 and with the blocks an SM has to run (0.72 us a chunk at the least, 0.25 and 0.55 for
// every block).  us per call, a thread per rollout / a warp per step: 2.0 / 2.4 for 2 x 32, 4.4 / 2.6 for 16 x 1024,
// 4.3 / 3.0 for 16 x 8192, 4.7 / 4.6 for 16 x 16384, 5.3 / 6.7 for 16 x 32768, 5.1 / 6.6 for 17 x 16384, 24.4 / 9.6 for
// 128 x 4096, 49 / 68 for 128 x 65536, 11.8 / 142 for 1 x 1048576.
bool thread_per_rollout(int n, int batch, bool discounts, int sm_count)
{
    const long long chunks = (n + kSteps - 1) / kSteps;
    const bool beyond_l2 = 4LL * n * batch * (discounts ? 5 : 4) > (64LL << 20);
    const long long step = (discounts ? 21 : 17) * (beyond_l2 ? 3 : 2) / 2;
    return step * n < chunks * std::max<long long>(72, 25 + 55LL * batch / (kCols * sm_count));
}

}  // namespace

}  // namespace accerl

using namespace accerl;

extern "C" accerl_status accerl_vtrace(const float *logp_smaller_dev, const float *logp_original_dev,
                                       const float *rewards_dev, const float *values_dev,
                                       const float *bootstrap_dev, const float *discounts_dev,
                                       int32_t n_steps, int32_t batch, float gamma, float rho_hat,
                                       float c_hat, float *vs_dev, float *adv_dev, void *cuda_stream)
{
    if (!logp_smaller_dev || !logp_original_dev || !rewards_dev || !values_dev || !bootstrap_dev || !vs_dev) {
        set_error("vtrace: null argument");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (n_steps < 1 || batch < 1 || (long long)n_steps * batch >= (1LL << 40)) {
        set_error("vtrace: n_steps and batch must be positive (and n_steps * batch below 2^40)");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (!(gamma >= 0.f) || !(rho_hat > 0.f) || !(c_hat > 0.f) || !isfinite(gamma) || isnan(rho_hat) || isnan(c_hat)) {
        set_error("vtrace: gamma must be finite and non-negative, rho_hat and c_hat positive");
        return ACCERL_ERR_INVALID_ARG;
    }
    const uintptr_t all = (uintptr_t)logp_smaller_dev | (uintptr_t)logp_original_dev | (uintptr_t)rewards_dev |
                          (uintptr_t)values_dev | (uintptr_t)bootstrap_dev | (uintptr_t)discounts_dev |
                          (uintptr_t)vs_dev | (uintptr_t)adv_dev;
    if (all & 3) {
        set_error("vtrace: misaligned pointer (4 bytes needed)");
        return ACCERL_ERR_INVALID_ARG;
    }
    int device = 0, sm_count = 0;
    ACCERL_CUDA_TRY(cudaGetDevice(&device));
    ACCERL_CUDA_TRY(cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, device));
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (thread_per_rollout(n_steps, batch, discounts_dev != nullptr, sm_count)) {
        const int threads = batch >= sm_count * 128 * 4 ? 128 : 32;  // few rollouts: spread them over the SMs
        vtrace_rollout_kernel<<<(unsigned)((batch + threads - 1) / threads), threads, 0, st>>>(
            logp_smaller_dev, logp_original_dev, rewards_dev, values_dev, bootstrap_dev, discounts_dev, n_steps,
            batch, gamma, rho_hat, c_hat, vs_dev, adv_dev);
    } else {
        vtrace_kernel<<<(unsigned)((batch + kCols - 1) / kCols), 32 * kSteps, 0, st>>>(
            logp_smaller_dev, logp_original_dev, rewards_dev, values_dev, bootstrap_dev, discounts_dev, n_steps,
            batch, gamma, rho_hat, c_hat, vs_dev, adv_dev);
    }
    ACCERL_CUDA_TRY(cudaGetLastError());
    return ACCERL_OK;
}
