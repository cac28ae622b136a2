// Single-fma requantiser: the search, at create, for the per-channel constants.
//
// The requantiser q(acc) = clamp(rintf(relu?(fmaf((float)acc, k, b)) / s_out), -128, 127) is a
// non-decreasing step function of the int32 accumulator (k = s_in * s_w[c] > 0; every rounding
// in it is monotone).  So is a(acc) = relu?(clamp(rint(fmaf((float)acc, k2, b2)))) for k2 > 0.
// Two non-decreasing functions that agree on every integer of [lo, hi], with both already at the
// lowest code at lo and at 127 at hi, agree on all of int32.  And they agree on [lo, hi] if they agree at
// its ends and rise to each code at the same integer.  So a thread finds the first accumulator of one
// code by bisection, and a candidate pair is compared there and one below: two evaluations a thread
// instead of the whole band of a few hundred thousand integers, with the same outcome for every
// candidate.  (k2, b2) = (fl(k / s_out),
// fl(b / s_out)) is right for most channels; where a handful of accumulators near a rounding tie
// come out differently, neighbours of the pair are tried -- b2 in steps of 2^-21, k2 in ulps --
// until one agrees everywhere.  A layer all of whose channels have such a pair runs its epilogue
// with one fma per element instead of the three-step division; any other layer keeps that one.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "epilogue.cuh"
#include "internal.h"
#include "tc_gemm.h"

namespace accerl {

namespace {

constexpr int kKOffsets = 25;   // k2: 0, +1, -1, ... +12, -12 ulps
constexpr int kBOffsets = 49;   // b2: 0, +1, -1, ... +24, -24 steps of 2^-21
constexpr int kFitThreads = 256;
constexpr int kFitGroup = 8;    // candidates compared between two votes

struct FitJob {
    float s_out;
    int relu;
    float k, b;          // the channel's epilogue constants
    float k0, b0;        // fl(k / s_out), fl(b / s_out)
    long long lo, hi;    // band of accumulators to compare (inside int32)
    int check_lo, check_hi;  // 1: the band's end is no int32 limit, so both functions must be saturated there
};

struct FitResult {
    float k2, b2;
    int found, tries;
};

__device__ __forceinline__ int alternate(int i) { return (i & 1) ? (i + 1) / 2 : -(i / 2); }  // 0, 1, -1, 2, -2, ...

// A block per channel, a thread per code above the band's lowest (at most 255).  Bound by the chain of
// votes over the candidates of a channel that has no pair at all (a few per wide fully connected layer).
// The 656 channels of a residual network: 597 us comparing whole bands, 239 us.
__global__ void __launch_bounds__(kFitThreads) fit_affine_kernel(const FitJob *jobs, FitResult *results)
{
    __shared__ unsigned failed[3];  // candidates of a group that some thread refutes, three groups in turn
    const FitJob job = jobs[blockIdx.x];
    const bool relu = job.relu != 0;
    auto code = [&](long long a) { return exact_code(epilogue_float((int)a, job.k, job.b, false), job.s_out, relu); };
    const int code_lo = code(job.lo), code_hi = code(job.hi), mine = code_lo + 1 + (int)threadIdx.x;
    if (threadIdx.x < 3) failed[threadIdx.x] = 0;
    // The first accumulator with this thread's code or a higher one; the thread behind the last code takes the
    // band's ends instead.
    const bool rises = mine <= code_hi, ends = mine == code_hi + 1;
    long long below = job.lo, first = job.hi;
    if (rises) {
        while (first - below > 1) {
            const long long mid = below + (first - below) / 2;
            if (code(mid) >= mine) first = mid;
            else below = mid;
        }
    }
    const float x0 = __int2float_rn((int)below), x1 = __int2float_rn((int)first);
    // saturated at an end that is no int32 limit
    const bool ends_ok = (!job.check_lo || code_lo == (relu ? 0 : -128)) && (!job.check_hi || code_hi == 127);
    auto refuted = [&](float k2, float b2) {
        const int a0 = affine_code(x0, k2, b2, relu), a1 = affine_code(x1, k2, b2, relu);
        return rises ? a0 >= mine || a1 < mine : ends && (!ends_ok || a0 != code_lo || a1 != code_hi);
    };
    auto candidate_k = [&](int cand) { return __uint_as_float(__float_as_uint(job.k0) + (unsigned)alternate(cand % kKOffsets)); };
    auto candidate_b = [&](int cand) { return __fadd_rn(job.b0, __int2float_rn(alternate(cand / kKOffsets)) * 4.76837158203125e-7f); };
    __syncthreads();
    constexpr int kCands = kKOffsets * kBOffsets;
    for (int cand0 = 0, group = 0; cand0 < kCands; cand0 += kFitGroup, group = group == 2 ? 0 : group + 1) {
        unsigned mask = 0;
#pragma unroll
        for (int j = 0; j < kFitGroup; ++j) {
            const float k2 = candidate_k(cand0 + j);
            if (cand0 + j >= kCands || !(k2 > 0.f) || refuted(k2, candidate_b(cand0 + j))) mask |= 1u << j;
        }
        mask = __reduce_or_sync(0xffffffffu, mask);
        if ((threadIdx.x & 31) == 0 && mask) atomicOr(&failed[group], mask);
        __syncthreads();
        const unsigned left = ~failed[group] & ((1u << kFitGroup) - 1);
        // (the group before was read before this vote and its word is written again after the next one)
        if (threadIdx.x == 0) failed[group == 0 ? 2 : group - 1] = 0;
        if (left) {
            const int cand = cand0 + __ffs(left) - 1;
            if (threadIdx.x == 0) results[blockIdx.x] = FitResult{candidate_k(cand), candidate_b(cand), 1, cand + 1};
            return;
        }
    }
    if (threadIdx.x == 0) results[blockIdx.x] = FitResult{job.k0, job.b0, 0, kCands};
}

// band of accumulators outside which both requantisers are saturated (or which int32 ends)
bool make_job(float k, float b, float s_out, bool relu, FitJob *job)
{
    if (!(k > 0.f) || !(s_out > 0.f) || !std::isfinite(k) || !std::isfinite(b) || !std::isfinite(s_out)) return false;
    const double dk = k, db = b, ds = s_out;
    const float k0 = (float)(dk / ds), b0 = (float)(db / ds);
    if (!(k0 > 0.f) || !std::isfinite(k0) || !std::isfinite(b0)) return false;
    // y = -2 s (ReLU: the code is 0 below) or -130 s at the low end, +130 s at the high end
    double lo = std::floor(((relu ? -2.0 : -130.0) * ds - db) / dk), hi = std::ceil((130.0 * ds - db) / dk);
    lo -= 16.0 + std::fabs(lo) * 0x1p-20;  // (float)acc is inexact above 2^24
    hi += 16.0 + std::fabs(hi) * 0x1p-20;
    job->s_out = s_out;
    job->relu = relu ? 1 : 0;
    job->k = k;
    job->b = b;
    job->k0 = k0;
    job->b0 = b0;
    job->check_lo = lo >= -2147483648.0;
    job->check_hi = hi <= 2147483647.0;
    job->lo = (long long)std::max(lo, -2147483648.0);
    job->hi = (long long)std::min(hi, 2147483647.0);
    // (bands of the networks here have 65 k - 350 k accumulators; the limit is from when the whole band was compared, and
    // channels with wider ones still divide)
    return job->hi >= job->lo && job->hi - job->lo <= (1LL << 22);
}

}  // namespace

// ---------------------------------------------------------------------------------------
// the three-step division: is it exact for this scale?
// ---------------------------------------------------------------------------------------
namespace {

struct DivJob {
    float s, r;
    unsigned lo, hi;  // bit patterns of the positive y to compare
};

// Positive y only (every operation of both sides is odd in y, and the clamp is applied to equal
// integers), and only from 0.4 s to 130 s: below, both quotients are far from 0.5 and round to 0; above,
// both are beyond 129 and saturate.  Some 70 million values instead of 2^32: 0.1 ms instead of 4.5.
__global__ void __launch_bounds__(256) verify_fastdiv_kernel(const DivJob *jobs, int *bad)
{
    const DivJob job = jobs[blockIdx.y];
    const unsigned stride = gridDim.x * blockDim.x;
    bool wrong = false;
    for (unsigned long long i = job.lo + (unsigned long long)(blockIdx.x * blockDim.x + threadIdx.x); i <= job.hi && !wrong; i += stride) {
        const float y = __uint_as_float((unsigned)i);
        wrong = fastdiv_rint(y, job.s, job.r) != __float2int_rn(__fdiv_rn(y, job.s));
    }
    if (wrong) bad[blockIdx.y] = 1;
}

struct DivKnown {
    float s, r;
    bool ok;
};
std::mutex g_div_mu;
std::vector<DivKnown> g_div_known;  // scales checked before, at most kDivKnown of them
constexpr size_t kDivKnown = 4096;

}  // namespace

// ---------------------------------------------------------------------------------------
// the requantisers of a whole network
// ---------------------------------------------------------------------------------------
// For every requantising layer: single-fma constants for all its channels, or a verified reciprocal for
// the three-step division, or neither.  One launch searches the channels of all layers and at most three
// more check the divisions of the layers the search left over (layer by layer, with an allocation, two
// copies and a launch each, this was most of the time a policy took to build).
accerl_status fit_requants(accerl_policy *p, const accerl_layer_desc *layers, int n_layers)
{
    if (!p->requant.empty()) return ACCERL_OK;
    std::vector<LayerRequant> rq(n_layers);
    std::vector<FitJob> jobs;
    std::vector<std::vector<int>> job_of(n_layers);
    for (int i = 0; i < n_layers; ++i) {
        const accerl_layer_desc &d = layers[i];
        if (d.kind == ACCERL_MAXPOOL) continue;
        LayerRequant &q = rq[i];
        q.k.resize(d.out_c);
        q.b.resize(d.out_c);
        for (int c = 0; c < d.out_c; ++c) {
            volatile float k = d.s_in * d.s_w[c];  // one fp32 rounding, never contracted
            q.k[c] = k;
            q.b[c] = d.bias[c];
        }
        volatile float inv = 1.0f / d.s_out;  // IEEE reciprocal, rounded once
        q.inv_s_out = inv;
        if ((d.flags & ACCERL_LOGITS) || (p->flags & (ACCERL_FLAG_TEST_NO_FASTDIV | ACCERL_FLAG_TEST_NO_AFFINE))) continue;
        std::vector<FitJob> mine(d.out_c);
        bool all = true;
        for (int c = 0; c < d.out_c && all; ++c)
            all = make_job(q.k[c], q.b[c], d.s_out, (d.flags & ACCERL_RELU_OUT) != 0, &mine[c]);
        if (!all) continue;
        for (const FitJob &j : mine) {
            job_of[i].push_back((int)jobs.size());
            jobs.push_back(j);
        }
    }
    struct Device {  // one block of device memory for both steps
        char *ptr = nullptr;
        ~Device()
        {
            // (where a call failed, its kernels may still run)
            if (ptr) device_free(ptr, cudaStreamSynchronize(0) == cudaSuccess);
        }
    } dev;
    const size_t job_bytes = (jobs.size() * sizeof(FitJob) + 255) / 256 * 256, res_bytes = (jobs.size() * sizeof(FitResult) + 255) / 256 * 256;
    const size_t div_bytes = ((size_t)n_layers * sizeof(DivJob) + 255) / 256 * 256;
    ACCERL_CUDA_TRY(device_alloc((void **)&dev.ptr, job_bytes + res_bytes + div_bytes + (size_t)n_layers * sizeof(int) + 256));
    if (!jobs.empty()) {
        std::vector<FitResult> res(jobs.size());
        ACCERL_CUDA_TRY(cudaMemcpyAsync(dev.ptr, jobs.data(), jobs.size() * sizeof(FitJob), cudaMemcpyHostToDevice, 0));
        fit_affine_kernel<<<(unsigned)jobs.size(), kFitThreads>>>((const FitJob *)dev.ptr, (FitResult *)(dev.ptr + job_bytes));
        ACCERL_CUDA_TRY(cudaGetLastError());
        ACCERL_CUDA_TRY(cudaMemcpy(res.data(), dev.ptr + job_bytes, res.size() * sizeof(FitResult), cudaMemcpyDeviceToHost));
        for (int i = 0; i < n_layers; ++i) {
            bool found = !job_of[i].empty();
            for (int j : job_of[i]) found = found && res[j].found;
            if (!found) continue;
            for (size_t c = 0; c < job_of[i].size(); ++c) {
                rq[i].k[c] = res[job_of[i][c]].k2;
                rq[i].b[c] = res[job_of[i][c]].b2;
            }
            rq[i].affine = rq[i].fast_div = 1;  // a verified division-free requantiser exists
        }
    }
    // fl(1 / s_out) or, where that one fails, one of its two neighbours (the correction step works with any
    // reciprocal that close; which rare operand patterns round wrongly differs between them)
    std::lock_guard<std::mutex> lock(g_div_mu);
    for (int cand = 0; cand < 3; ++cand) {
        std::vector<DivJob> div;
        std::vector<int> of;
        auto settle = [&](int i, float r, bool ok) {
            if (ok) {
                rq[i].fast_div = 1;
                rq[i].inv_s_out = r;
            }
        };
        for (int i = 0; i < n_layers; ++i) {
            const accerl_layer_desc &d = layers[i];
            if (d.kind == ACCERL_MAXPOOL || (d.flags & ACCERL_LOGITS) || rq[i].fast_div || (p->flags & ACCERL_FLAG_TEST_NO_FASTDIV)) continue;
            // scales for which a quotient of the largest |y| (|acc| < 2^31) or a correction term could leave
            // the normal range are not considered
            float kmax = 0.f, bmax = 0.f;
            for (size_t c = 0; c < rq[i].k.size(); ++c) {
                kmax = std::max(kmax, rq[i].k[c]);
                bmax = std::max(bmax, std::fabs(rq[i].b[c]));
            }
            const double y_max = 2147483648.0 * kmax + bmax;
            if (!(d.s_out > 1e-25f && d.s_out < 1e25f && y_max < 1e30 && y_max / d.s_out < 1e30)) continue;
            const float r0 = rq[i].inv_s_out, r = cand == 0 ? r0 : (cand == 1 ? std::nextafter(r0, 2.f * r0) : std::nextafter(r0, 0.f));
            bool known = false;
            for (const DivKnown &k : g_div_known)
                if (k.s == d.s_out && k.r == r) {
                    settle(i, r, k.ok);
                    known = true;
                }
            if (known) continue;
            DivJob j;
            const float lo = 0.4f * d.s_out, hi = 130.f * d.s_out;
            j.s = d.s_out;
            j.r = r;
            memcpy(&j.lo, &lo, 4);
            memcpy(&j.hi, &hi, 4);
            div.push_back(j);
            of.push_back(i);
        }
        if (div.empty()) continue;
        char *d_div = dev.ptr + job_bytes + res_bytes;
        int *d_bad = (int *)(d_div + div_bytes);
        std::vector<int> bad(div.size());
        ACCERL_CUDA_TRY(cudaMemcpyAsync(d_div, div.data(), div.size() * sizeof(DivJob), cudaMemcpyHostToDevice, 0));
        ACCERL_CUDA_TRY(cudaMemsetAsync(d_bad, 0, div.size() * sizeof(int), 0));
        verify_fastdiv_kernel<<<dim3(148 * 2, (unsigned)div.size()), 256>>>((const DivJob *)d_div, d_bad);
        ACCERL_CUDA_TRY(cudaGetLastError());
        ACCERL_CUDA_TRY(cudaMemcpy(bad.data(), d_bad, bad.size() * sizeof(int), cudaMemcpyDeviceToHost));
        if (g_div_known.size() + div.size() > kDivKnown) g_div_known.clear();
        for (size_t j = 0; j < div.size(); ++j) {
            g_div_known.push_back(DivKnown{div[j].s, div[j].r, bad[j] == 0});
            settle(of[j], div[j].r, bad[j] == 0);
        }
    }
    p->requant = std::move(rq);
    return ACCERL_OK;
}

}  // namespace accerl
