// The sampler of the launches that end in a row of logits per warp.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace accerl {

// One row per warp, one lane per action: the arithmetic of sample_warp_kernel for a full-warp
// segment.  Every lane returns the drawn action and its log-prob.
template <bool ENTROPY>
__device__ __forceinline__ void warp_sample(float z, bool live, float uu, int A, int lane, int &a,
                                            float &lpa, float &h)
{
    if (!live) z = -INFINITY;
    float m = z;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    // the first maximal lane contributes exp(0) = 1 exactly: sum the others, take log1p
    const unsigned ismax = __ballot_sync(0xffffffffu, live && z == m);
    const int amax = ismax ? __ffs(ismax) - 1 : 0;
    float s = (live && lane != amax) ? expf(z - m) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float lp = live ? (z - m) - log1pf(s) : 0.f;
    float cdf = live ? expf(lp) : 0.f;  // inclusive scan
    if (ENTROPY) {  // H = -sum p log p
        h = cdf > 0.f ? -cdf * lp : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float v = __shfl_up_sync(0xffffffffu, cdf, o);
        if (lane >= o) cdf += v;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, live && uu < cdf);
    a = hit ? __ffs(hit) - 1 : A - 1;
    lpa = __shfl_sync(0xffffffffu, lp, a);
}

}  // namespace accerl
