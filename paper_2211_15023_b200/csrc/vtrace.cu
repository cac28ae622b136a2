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

#include "internal.h"

namespace accerl {

namespace {

constexpr int kCols = 32;   // rollouts of a block, one per lane
constexpr int kSteps = 16;  // time steps of a chunk, one warp each

// The recursion is sequential in t, but only two multiply-adds a step of it: the ratios (an exp),
// the temporal differences and the advantages of all steps are independent.  So a block takes 32
// rollouts and, from the last step backwards, 16 steps at a time: warp w loads step w of the chunk
// (whole lines: arrays are time-major) and computes rho, g c and delta, the first warp runs the
// recursion over the chunk out of shared memory, and every warp writes its step's results.  The next
// chunk's loads are issued before the recursion of the current one.  With one thread per rollout and
// loads eight steps ahead the kernel was a chain of exps and memory latencies (6.1 us a call for 16 x 8192,
// now about 4).
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
    vtrace_kernel<<<(unsigned)((batch + kCols - 1) / kCols), 32 * kSteps, 0, (cudaStream_t)cuda_stream>>>(
        logp_smaller_dev, logp_original_dev, rewards_dev, values_dev, bootstrap_dev, discounts_dev, n_steps,
        batch, gamma, rho_hat, c_hat, vs_dev, adv_dev);
    ACCERL_CUDA_TRY(cudaGetLastError());
    return ACCERL_OK;
}
