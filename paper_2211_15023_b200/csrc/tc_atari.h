// Parameters of the image-resident kernel of the Atari conv stacks (tc_atari.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace accerl {

// Which states of a batch a launch works on: all `batch` of them in order, or, with `count`, the *count
// states listed in `rows` (both written on the device, see accerl_policy_act_mixed; *count <= batch).
// Intermediate tensors are compact (entry i belongs to state rows[i]).
struct Route {
    const int *rows = nullptr, *count = nullptr;
    int expect = 0;  // the caller's guess of *count, for choosing launch shapes
};
#ifdef __CUDACC__
// (call after griddepcontrol.wait)
__device__ __forceinline__ int routed_batch(const Route &r, int batch) { return r.count ? __ldcg(r.count) : batch; }
__device__ __forceinline__ int routed_row(const Route &r, int i) { return r.rows ? __ldcg(r.rows + i) : i; }
#endif

struct AtariLayer {
    float k[64], b[64];  // per channel: the single-fma pair, or (s_in * s_w, bias) for the division
    float s_out, inv_s_out;
    int affine, relu;
};

// 84 x 84 x 4 frames -> conv 8 x 8 / 4 -> 20 x 20 -> conv 4 x 4 / 2 -> 9 x 9 -> conv 3 x 3 -> 7 x 7, with
// 32 / 64 / 64 or 16 / 32 / 32 channels
struct AtariParams {
    const uint8_t *obs, *w;  // w: the three layers' weights in the kernel's layout
    int8_t *out;             // [n][49 * C3]: the fc layer's input rows
    int8_t *tap1, *tap2;     // outputs of the first two convs as the launch-per-layer plan stores them, or null
    int batch, wide;         // wide: 32 / 64 / 64 channels
    Route route;
    int ingest_mode;         // 2: u >> 1, 1: line with the minimum, 0: line without
    uint32_t ingest_mul, ingest_add;
    int *status;
    AtariLayer layer[3];
};

static_assert(sizeof(AtariLayer) % 16 == 0 && offsetof(AtariParams, layer) % 16 == 0, "constants are read 16 bytes at a time");

constexpr int kAtariWeightsWide = 4 * 32 * 64 + 4 * 64 * 128 + 9 * 64 * 64, kAtariWeightsNarrow = 4 * 16 * 64 + 4 * 32 * 64 + 9 * 32 * 32;

cudaError_t atari_launch(const AtariParams &p, int sm_count, cudaStream_t st);

}  // namespace accerl
