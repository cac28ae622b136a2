// The Monitor's indicators and the per-state choice between two policies (Section 2.4).
//
// kl_rows_kernel / kl_wide_kernel: KL(pi_original || pi_smaller) per state from two logit matrices
// (Eq. KL), a thread or a warp per state; kl_stats_kernel reduces the per-state values to their mean and
// maximum (the "KL mean" and "KL max" indicators) in one CTA or one cluster of CTAs, in a fixed order, so
// that the result does not depend on scheduling.  route_kernel lists the states of each network for
// the linear-alpha strategy of Section 3.2 (the Actor follows the small network where the selector draw falls
// below alpha), so that each runs on its own states only; where a plan cannot do that, both run on all of them and
// mix_select_kernel overwrites the original policy's outputs with the smaller policy's.
#include <cooperative_groups.h>
#include <math.h>

#include "internal.h"

namespace accerl {

namespace {

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_maxf(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Double arithmetic: where the two policies nearly agree the terms p (log p - log q) cancel, and
// the indicator runs at the Monitor's interval, not per environment step.  With e_i = exp(zo_i - mo),
//   KL = sum_i e_i / so (zo_i - zs_i) - (lse_o - lse_s),
// two exponentials an action instead of three, and identical rows give exactly 0.

// exp(x) for x <= 0 by table and a short polynomial (Tang, "Table-driven implementation of the exponential
// function", 1989): x = (64 m + j) ln2 / 64 + r, |r| <= ln2 / 128, exp(x) = 2^m 2^(j/64) (1 + r + ... + r^5 / 120);
// the truncation is below 3e-17, the result within about one ulp.  `table` holds 2^(j/64).  It has half the
// instructions of exp(), of which the rows kernel needs two per action (16 x 8192 rollouts of 18 actions,
// V-trace and both launches of the KL, rows copied element by element as they were then: 27 us with exp(), 24.6 with this).
__device__ __forceinline__ double exp_nonpositive(double x, const double *table)
{
    const double shift = 6755399441055744.0;  // 1.5 * 2^52: adding it rounds to an integer
    const double t = fma(x, 92.332482616893656, shift), nf = t - shift;
    const int n = __double2loint(t);
    const double r = fma(nf, -3.623510646634843e-19, fma(nf, -0.010830424696249145, x));
    const double p = fma(r * r, fma(r, fma(r, fma(r, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5), r);
    const double v = fma(table[n & 63], p, table[n & 63]);
    const double y = __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
    // What underflows is nothing beside the row's largest term; the last case is a NaN.
    return x >= -708.0 ? y : x < 0.0 ? 0.0 : x;
}

// One row by one thread, V elements a load (then the row's address is a multiple of V elements and A one of V);
// the elements are added in order whatever V is.
template <int V>
__device__ __forceinline__ float kl_of_row(const float *zo, const float *zs, int A, const double *table)
{
    struct alignas(4 * V) Piece {
        float v[V];
    };
    const Piece *po = reinterpret_cast<const Piece *>(zo), *ps = reinterpret_cast<const Piece *>(zs);
    const int pieces = A / V;
    float fo = zo[0], fs = zs[0];
    for (int i = 0; i < pieces; ++i) {
        const Piece a = po[i], b = ps[i];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            fo = fmaxf(fo, a.v[k]);
            fs = fmaxf(fs, b.v[k]);
        }
    }
    const double mo = fo, ms = fs;
    double so = 0.0, ss = 0.0, acc = 0.0;
    for (int i = 0; i < pieces; ++i) {
        const Piece a = po[i], b = ps[i];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const double o = a.v[k], t = b.v[k], e = exp_nonpositive(o - mo, table);
            so += e;
            ss += exp_nonpositive(t - ms, table);
            if (e > 0.0) acc += e * (o - t);
        }
    }
    return (float)(acc / so - ((mo + log(so)) - (ms + log(ss))));
}

constexpr int kKlRows = 128;   // rows (and threads) of a block
constexpr int kKlCluster = 8;  // CTAs that share the reduction to mean and maximum

// The first thing of a kernel that ends in cluster_stats: this CTA's shared memory may be written from now on.
__device__ __forceinline__ void cluster_started() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }

// Mean and maximum over all threads of a cluster (every CTA calls with its own partial sum and
// maximum), or of one CTA; always the same order of additions.
template <bool CLUSTER>
__device__ __forceinline__ void cluster_stats(double sum, float mx, int B, float *stats)
{
    __shared__ double s_sum[32];
    __shared__ float s_max[32];
    __shared__ double c_sum[kKlCluster];  // used in the first CTA
    __shared__ float c_max[kKlCluster];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    sum = warp_sum(sum);
    mx = warp_maxf(mx);
    if (lane == 0) {
        s_sum[warp] = sum;
        s_max[warp] = mx;
    }
    __syncthreads();
    if (warp == 0) {
        sum = warp_sum(lane < warps ? s_sum[lane] : 0.0);
        mx = warp_maxf(lane < warps ? s_max[lane] : -INFINITY);
    }
    if (!CLUSTER) {
        if (threadIdx.x == 0) {
            stats[0] = (float)(sum / (double)B);
            stats[1] = mx;
        }
        return;
    }
    // The first CTA's shared memory exists only once that CTA has started (the arrivals of cluster_started lie a
    // whole pass over the rows back: nothing waits here)
    asm volatile("barrier.cluster.wait;" ::: "memory");
    if (threadIdx.x == 0) {
        const unsigned rank = cooperative_groups::this_cluster().block_rank();
        *cooperative_groups::this_cluster().map_shared_rank(&c_sum[rank], 0) = sum;
        *cooperative_groups::this_cluster().map_shared_rank(&c_max[rank], 0) = mx;
    }
    cooperative_groups::this_cluster().sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned n = cooperative_groups::this_cluster().num_blocks();
        sum = 0.0;
        mx = -INFINITY;
        for (unsigned i = 0; i < n; ++i) {
            sum += c_sum[i];
            mx = fmaxf(mx, c_max[i]);
        }
        stats[0] = (float)(sum / (double)B);
        stats[1] = mx;
    }
}

// Many rows of at most 64 actions, or few of at most 12 (see the choice in accerl_policy_kl): one thread per
// row.  A block's rows are contiguous in memory; they pass through shared memory, by asynchronous copies that
// are all in flight at once, so that the loads are whole lines and every thread then walks its own row, a chain
// of two exponentials an action.  A warp per row, as below, leaves 14 of 32 lanes idle at 18 actions and spends
// its time in shuffles; with that and a one-block reduction the two launches for 131072 rows of 18 took 119 us,
// with this kernel 20.7 element by element and 18.7 in 16-byte copies (with V-trace 24.6 and 22.6; rows of 9 actions 16.5
// and 14.5, of 31 26.8 and 24.7, of 62 51.1 and 43.2).
//
// V > 0: the rows lie in shared memory as in global memory and come in 16-byte copies (a fourth of the
// instructions, and no row and column to keep); a thread reads V = 1, 2 or 4 elements at a time, the width at which
// rows of that many elements fall into different banks.  V = 0, for rows of a multiple of eight elements,
// addresses that are none of 16 bytes and always with STATS: element by element into rows of an odd pitch.
//
// STATS (one cluster, at most kKlCluster blocks' rows a pass): the mean and the maximum come out of the same launch.
template <bool STATS, int V>
__global__ void __launch_bounds__(kKlRows)
kl_rows_kernel(const float *__restrict__ zo, const float *__restrict__ zs, int B, int A, int pitch,
               float *__restrict__ kl, float *__restrict__ stats)
{
    extern __shared__ __align__(16) float s_rows[];  // [2][kKlRows][pitch]
    __shared__ double s_table[64];
    if (STATS) cluster_started();
    if (threadIdx.x < 64) s_table[threadIdx.x] = exp2((double)threadIdx.x * (1.0 / 64.0));
    double sum = 0.0;
    float mx = -INFINITY;
    for (long long row0 = (long long)blockIdx.x * kKlRows; row0 < B; row0 += (long long)gridDim.x * kKlRows) {
        const int rows = (int)min((long long)kKlRows, B - row0), n = rows * A;
        const float *src[2] = {zo + row0 * A, zs + row0 * A};
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_rows), dst1 = dst + 4 * kKlRows * pitch;
        if constexpr (V > 0) {
            for (int i = 4 * threadIdx.x; i + 3 < n; i += 4 * kKlRows) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 4 * i), "l"(src[0] + i) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst1 + 4 * i), "l"(src[1] + i) : "memory");
            }
            if (const int i = (n & ~3) + (int)threadIdx.x; i < n) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * i), "l"(src[0] + i) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst1 + 4 * i), "l"(src[1] + i) : "memory");
            }
        } else {
            int r = (int)threadIdx.x / A, c = (int)threadIdx.x - r * A;
            const int dr = kKlRows / A, dc = kKlRows - dr * A;
            for (int i = threadIdx.x; i < n; i += kKlRows) {
                const uint32_t d = 4 * (r * pitch + c);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + d), "l"(src[0] + i) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst1 + d), "l"(src[1] + i) : "memory");
                r += dr;
                c += dc;
                if (c >= A) {
                    c -= A;
                    ++r;
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if ((int)threadIdx.x < rows) {
            const float v = kl_of_row<V ? V : 1>(s_rows + threadIdx.x * pitch, s_rows + (kKlRows + threadIdx.x) * pitch, A, s_table);
            kl[row0 + threadIdx.x] = v;
            sum += (double)v;
            mx = fmaxf(mx, v);
        }
        __syncthreads();
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (STATS) cluster_stats<true>(sum, mx, B, stats);
}

// any A: one warp per row, lanes striding over the actions (a row's chain is short: what few rows need)
__global__ void __launch_bounds__(128)
kl_wide_kernel(const float *__restrict__ zo_all, const float *__restrict__ zs_all, int B, int A,
               float *__restrict__ kl)
{
    const int lane = threadIdx.x & 31;
    const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= B) return;
    const float *zo = zo_all + row * A, *zs = zs_all + row * A;
    double mo = -INFINITY, ms = -INFINITY;
    for (int i = lane; i < A; i += 32) {
        mo = fmax(mo, (double)zo[i]);
        ms = fmax(ms, (double)zs[i]);
    }
    mo = warp_max(mo);
    ms = warp_max(ms);
    double so = 0.0, ss = 0.0, acc = 0.0;
    for (int i = lane; i < A; i += 32) {
        const double o = zo[i], s = zs[i], e = exp(o - mo);
        so += e;
        ss += exp(s - ms);
        if (e > 0.0) acc += e * (o - s);
    }
    so = warp_sum(so);
    ss = warp_sum(ss);
    acc = warp_sum(acc);
    if (lane == 0) kl[row] = (float)(acc / so - ((mo + log(so)) - (ms + log(ss))));
}

// stats[0] = mean, stats[1] = max of kl[0..B): one cluster, or for kOneCta rows at most one CTA, whose threads then
// have all their loads in flight at once (us per call, rows kernel included, one CTA / cluster of eight: 160 x 18
// 4.3 / 5.0, 1024 x 18 5.3 / 6.0, 4096 x 64 7.4 / 7.9, 8192 x 64 10.6 / 10.6, 12000 x 64 14.3 / 13.3)
constexpr int kOneCta = 8192;
template <bool CLUSTER>
__global__ void __launch_bounds__(1024) kl_stats_kernel(const float *__restrict__ kl, int B, float *stats)
{
    if (CLUSTER) cluster_started();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double sum = 0.0;
    float mx = -INFINITY;
    const long long stride = (long long)gridDim.x * blockDim.x;
    constexpr int kAhead = 8;  // loads in flight per thread: the kernel is a chain of memory latencies
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < B; i += kAhead * stride) {
        float v[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) v[j] = i + j * stride < B ? __ldcg(kl + i + j * stride) : -INFINITY;
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            if (i + j * stride < B) sum += (double)v[j];
            mx = fmaxf(mx, v[j]);
        }
    }
    cluster_stats<CLUSTER>(sum, mx, B, stats);
}

struct MixOut {
    float *logits;
    int32_t *actions;
    float *logp, *value, *entropy;
};

__global__ void __launch_bounds__(256)
mix_select_kernel(const float *__restrict__ u_select, float alpha, int B, int A, MixOut dst, MixOut src,
                  uint8_t *__restrict__ use_smaller)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const bool pick = u_select[b] < alpha;
    if (use_smaller) use_smaller[b] = pick ? 1 : 0;
    if (!pick) return;
    for (int i = 0; i < A; ++i) dst.logits[(long long)b * A + i] = src.logits[(long long)b * A + i];
    dst.actions[b] = src.actions[b];
    dst.logp[b] = src.logp[b];
    if (dst.value) dst.value[b] = src.value[b];
    if (dst.entropy) dst.entropy[b] = src.entropy[b];
}

// The states of each network, in order: rows[0 .. max) for the smaller one, rows[max .. 2 max) for the
// original, their counts behind.  One block: the lists must be complete before anything starts anyway.
constexpr int kRouteThreads = 1024;
__global__ void __launch_bounds__(kRouteThreads)
route_kernel(const float *__restrict__ u_select, float alpha, int B, int max_batch, int *__restrict__ rows,
             uint8_t *__restrict__ use_smaller)
{
    __shared__ int warp_base[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int base = 0;  // states of the smaller network before this pass
    for (int b0 = 0; b0 < B; b0 += kRouteThreads) {
        const int b = b0 + (int)threadIdx.x;
        const bool pick = b < B && u_select[b] < alpha;
        const unsigned mask = __ballot_sync(0xffffffffu, pick);
        if (lane == 0) warp_base[warp] = __popc(mask);
        __syncthreads();
        const int mine = warp_base[lane];
        int sum = mine;  // inclusive scan over the warps, by every warp for itself
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        const int before = base + __shfl_sync(0xffffffffu, sum - mine, warp) + __popc(mask & ((1u << lane) - 1));
        if (b < B) {
            if (pick) rows[before] = b;
            else rows[max_batch + b - before] = b;
            if (use_smaller) use_smaller[b] = pick ? 1 : 0;
        }
        base += __shfl_sync(0xffffffffu, sum, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        rows[2 * max_batch] = base;
        rows[2 * max_batch + 1] = B - base;
    }
}

}  // namespace

}  // namespace accerl

using namespace accerl;

extern "C" accerl_status accerl_policy_kl(const float *logits_original_dev, const float *logits_smaller_dev,
                                          int32_t batch, int32_t n_actions, float *kl_dev,
                                          float *kl_mean_max_dev, void *cuda_stream)
{
    if (!logits_original_dev || !logits_smaller_dev || !kl_dev) {
        set_error("kl: null argument");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (batch < 1 || n_actions < 1 || n_actions > 1024) {
        set_error("kl: batch must be positive and n_actions in 1..1024");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (((uintptr_t)logits_original_dev | (uintptr_t)logits_smaller_dev | (uintptr_t)kl_dev |
         (uintptr_t)kl_mean_max_dev) & 3) {
        set_error("kl: misaligned pointer (4 bytes needed)");
        return ACCERL_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // A thread per row pays from some 256 rows an action on, where a warp per row no longer fits the chip at once
    // (us per call, thread / warp: 18 actions 8.2 / 5.6 for 2048 rows, 8.2 / 8.4 for 6144, 9.7 / 22.7 for 32768; 64
    // actions 15.1 / 6.0, 15.3 / 9.1, 18.3 / 27).  Few short rows go to one cluster that does it all, in a second
    // pass only where they are shorter still: a second launch costs some 2 us, what a pass over 1024 rows takes at 9
    // actions (9 actions: 4.4 for 1024 rows, 6.6 for 2048, the two launches 5.2 and 5.6).
    const long long rows_blocks = ((long long)batch + kKlRows - 1) / kKlRows;
    const bool one_launch = kl_mean_max_dev && n_actions <= 12 && rows_blocks <= (n_actions <= 6 ? 2 : 1) * kKlCluster;
    const bool narrow = n_actions <= 64 && (one_launch || batch >= 256 * n_actions);  // (66 KB of shared memory at 64)
    const bool whole = !one_launch && n_actions % 8 != 0 && (((uintptr_t)logits_original_dev | (uintptr_t)logits_smaller_dev) & 15) == 0;
    const int pitch = whole ? n_actions : n_actions | 1;
    const size_t smem = 2 * sizeof(float) * (size_t)kKlRows * pitch;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.stream = st;
    cfg.attrs = attr;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    const long long blocks = narrow ? rows_blocks : ((long long)batch * 32 + 127) / 128;
    if (one_launch) {
        const unsigned n = (unsigned)(blocks < kKlCluster ? blocks : kKlCluster);
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(kKlRows);
        cfg.dynamicSmemBytes = smem;
        attr[0].val.clusterDim.x = n;
        cfg.numAttrs = 1;
        ACCERL_CUDA_TRY(allow_smem((const void *)kl_rows_kernel<true, 0>, smem));
        ACCERL_CUDA_TRY(cudaLaunchKernelEx(&cfg, kl_rows_kernel<true, 0>, logits_original_dev, logits_smaller_dev, batch,
                                           n_actions, pitch, kl_dev, kl_mean_max_dev));
        return ACCERL_OK;
    }
    if (narrow) {
        const auto kernel = !whole ? kl_rows_kernel<false, 0>
                                   : n_actions % 2 ? kl_rows_kernel<false, 1> : n_actions % 4 ? kl_rows_kernel<false, 2> : kl_rows_kernel<false, 4>;
        ACCERL_CUDA_TRY(allow_smem((const void *)kernel, smem));
        kernel<<<(unsigned)blocks, kKlRows, smem, st>>>(logits_original_dev, logits_smaller_dev, batch, n_actions, pitch, kl_dev, nullptr);
    } else {
        kl_wide_kernel<<<(unsigned)blocks, 128, 0, st>>>(logits_original_dev, logits_smaller_dev, batch, n_actions, kl_dev);
    }
    ACCERL_CUDA_TRY(cudaGetLastError());
    if (kl_mean_max_dev) {
        const bool one = batch <= kOneCta;
        cfg.gridDim = dim3(one ? 1 : kKlCluster);
        cfg.blockDim = dim3(1024);
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = kKlCluster;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = one ? 1 : 2;
        ACCERL_CUDA_TRY(cudaLaunchKernelEx(&cfg, one ? kl_stats_kernel<false> : kl_stats_kernel<true>, (const float *)kl_dev, batch,
                                           kl_mean_max_dev));
    }
    return ACCERL_OK;
}

extern "C" accerl_status accerl_policy_act_mixed(accerl_policy *smaller, accerl_policy *original,
                                                 const void *obs_dev, const float *uniforms_dev,
                                                 const float *select_uniforms_dev, float alpha,
                                                 int32_t batch, float *logits_dev, int32_t *actions_dev,
                                                 float *logp_dev, float *value_dev, float *entropy_dev,
                                                 uint8_t *use_smaller_dev, void *cuda_stream)
{
    if (!smaller || !original || !select_uniforms_dev) {
        set_error("act_mixed: null argument");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (smaller == original) {
        set_error("act_mixed: the two handles must differ (each owns the workspace its kernels write)");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (smaller->n_actions != original->n_actions || smaller->device != original->device ||
        smaller->in_kind != original->in_kind || smaller->in_c != original->in_c ||
        smaller->in_h != original->in_h || smaller->in_w != original->in_w) {
        set_error("act_mixed: the two policies must share device, observation shape and action count");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (!(alpha >= 0.f && alpha <= 1.f)) {
        set_error("act_mixed: alpha must lie in [0, 1]");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (batch < 1 || batch > smaller->max_batch || batch > original->max_batch) {
        set_error("act_mixed: batch %d outside 1..min(max_batch) = %d", batch,
                  smaller->max_batch < original->max_batch ? smaller->max_batch : original->max_batch);
        return batch < 1 ? ACCERL_ERR_INVALID_ARG : ACCERL_ERR_BATCH_TOO_LARGE;
    }
    if (value_dev && (smaller->n_out == smaller->n_actions || original->n_out == original->n_actions)) {
        set_error("act_mixed: value_dev given but a handle was created without ACCERL_FLAG_VALUE_HEAD");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (((uintptr_t)select_uniforms_dev & 3)) {
        set_error("act_mixed: misaligned pointer");
        return ACCERL_ERR_INVALID_ARG;
    }
    int prev = -1;
    if (cudaGetDevice(&prev) == cudaSuccess && prev == smaller->device) prev = -1;
    else ACCERL_CUDA_TRY(cudaSetDevice(smaller->device));
    struct Restore {
        int prev;
        ~Restore() { if (prev >= 0) cudaSetDevice(prev); }
    } restore{prev};
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (!smaller->routed_steps.empty() && !original->routed_steps.empty()) {
        // Every state runs through its own network only: the states are listed per network, the first
        // launches gather by those lists, everything between is compact, the last launches scatter.
        // (Both networks on the whole batch: 2048 states of student and Nature-CNN, alpha 0.8, 123 us; so
        // 77.)  The numbers of states stay on the device; alpha tells the host what to expect.
        if (((uintptr_t)obs_dev & 15) || (((uintptr_t)uniforms_dev | (uintptr_t)logits_dev | (uintptr_t)actions_dev | (uintptr_t)logp_dev |
                                           (uintptr_t)value_dev | (uintptr_t)entropy_dev) & 3)) {
            set_error("act_mixed: misaligned pointer (obs needs 16 bytes, the others 4)");
            return ACCERL_ERR_INVALID_ARG;
        }
        if (!obs_dev || !uniforms_dev || !logits_dev || !actions_dev || !logp_dev) {
            set_error("act_mixed: null argument");
            return ACCERL_ERR_INVALID_ARG;
        }
        const int mb = smaller->max_batch;
        if (!smaller->mix_rows) {
            void *d = nullptr;
            const size_t bytes = sizeof(int) * (2 * (size_t)mb + 2) + 256;
            ACCERL_CUDA_TRY(device_alloc(&d, bytes));
            smaller->owned.push_back(d);
            smaller->workspace_bytes += bytes;
            smaller->mix_rows = (int *)d;
        }
        int *rows = smaller->mix_rows;
        route_kernel<<<1, kRouteThreads, 0, st>>>(select_uniforms_dev, alpha, batch, mb, rows, use_smaller_dev);
        ACCERL_CUDA_TRY(cudaGetLastError());
        // The two networks share nothing but the lists: side by side on two streams their small launches
        // fill each other's gaps (one after the other: 88 us for the case above).
        if (!smaller->mix.stream) ACCERL_CUDA_TRY(take_side_stream(&smaller->mix));
        SideWork side(st, smaller->mix);
        ACCERL_CUDA_TRY(side.begin());
        accerl_status result = ACCERL_OK;
        for (int i = 1; i >= 0; --i) {
            Route r;
            r.rows = rows + (size_t)i * mb;
            r.count = rows + 2 * (size_t)mb + i;
            r.expect = (int)ceilf((float)batch * (i ? 1.f - alpha : alpha));
            accerl_status s = run_steps(i ? original : smaller, obs_dev, uniforms_dev, batch, logits_dev, actions_dev, logp_dev,
                                        value_dev, entropy_dev, i ? st : smaller->mix.stream, nullptr, r);
            if (result == ACCERL_OK) result = s;
        }
        smaller->last_stream = st;  // (which waits for the other)
        if (result != ACCERL_OK) return result;
        ACCERL_CUDA_TRY(side.join());
        return ACCERL_OK;
    }
    // the original policy writes the caller's buffers, the smaller one the handle's own
    accerl_status s = accerl_policy_act_ex(original, obs_dev, uniforms_dev, batch, logits_dev, actions_dev,
                                           logp_dev, value_dev, entropy_dev, cuda_stream);
    if (s != ACCERL_OK) return s;
    if (!smaller->mix_logits) {
        const size_t mb = (size_t)smaller->max_batch;
        const size_t sz[5] = {4 * mb * (size_t)smaller->n_actions, 4 * mb, 4 * mb, 4 * mb, 4 * mb};
        void *d[5];
        for (int i = 0; i < 5; ++i) {
            ACCERL_CUDA_TRY(device_alloc(&d[i], sz[i] + 256));
            smaller->owned.push_back(d[i]);
            smaller->workspace_bytes += sz[i] + 256;
        }
        smaller->mix_actions = (int32_t *)d[1];
        smaller->mix_logp = (float *)d[2];
        smaller->mix_value = (float *)d[3];
        smaller->mix_entropy = (float *)d[4];
        smaller->mix_logits = (float *)d[0];
    }
    s = accerl_policy_act_ex(smaller, obs_dev, uniforms_dev, batch, smaller->mix_logits, smaller->mix_actions,
                             smaller->mix_logp, value_dev ? smaller->mix_value : nullptr,
                             entropy_dev ? smaller->mix_entropy : nullptr, cuda_stream);
    if (s != ACCERL_OK) return s;
    MixOut dst{logits_dev, actions_dev, logp_dev, value_dev, entropy_dev};
    MixOut src{smaller->mix_logits, smaller->mix_actions, smaller->mix_logp, smaller->mix_value,
               smaller->mix_entropy};
    mix_select_kernel<<<(unsigned)((batch + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        select_uniforms_dev, alpha, batch, smaller->n_actions, dst, src, use_smaller_dev);
    ACCERL_CUDA_TRY(cudaGetLastError());
    return ACCERL_OK;
}
