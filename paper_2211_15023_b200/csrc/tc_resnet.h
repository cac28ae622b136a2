// Parameters of the image-resident kernels of the IMPALA residual network (tc_resnet.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "tc_atari.h"

namespace accerl {

// Requantisation constants of one conv layer, read from the constant bank 16 bytes at a time: in the kernels'
// parameters they lie at multiples of 16 bytes.
struct ResLayer {
    float k[32], b[32];  // per channel: the single-fma pair, or (s_in * s_w, bias) for the division
    uint32_t mul[32];    // residual multiplier in the 16-bit lane dp2a reads: skip_mul << (16 * (c & 1))
    float s_out, inv_s_out;
    int affine, pad;     // (a multiple of 16 bytes)
};

// Geometry: 84 x 84 frames, stacks of 41 x 41 x 16, 20 x 20 x 32 and 9 x 9 x 32.  Every tensor is a
// sequence of 32-byte rows (the operand rows of the MMAs), image lines W + 1 pixels apart: the zero
// pixel in front of a line is also the one behind the line before it.  One zero line above and below.
constexpr int kRes1Rows = 43 * 21, kRes2Rows = 22 * 21;        // stored rows of an image
constexpr int kRes1Bytes = kRes1Rows * 32, kRes2Bytes = kRes2Rows * 32;
constexpr int kRes3Bytes = 81 * 32;                            // plain, the fc layer's input row
constexpr int kResFirstWeights = 3 * 80 * 32;                  // first conv: 3 K steps of 80 columns
constexpr int kRes1Weights = 6 * 6 * 32 * 32;                  // four 16 -> 16 convs, two halves of 16 -> 32
constexpr int kRes2Weights = 9 * 9 * 32 * 32;                  // nine 32 -> 32 convs

struct ResFirstParams {  // frames -> first conv -> max-pool
    const uint8_t *obs, *w;
    int8_t *x1;               // [n][kRes1Bytes]
    int8_t *tap_in, *tap_x1;  // plain NHWC copies for the parity taps, or null
    int batch, ingest_mode;   // 2: u >> 1, else the fixed-point line
    Route route;
    uint32_t ingest_mul, ingest_add;
    int *status;
    uint64_t pad = 0;
    ResLayer layer;
};

struct ResStack1Params {  // two residual blocks at 41 x 41, conv 16 -> 32, max-pool
    const int8_t *x1;
    const uint8_t *w;
    int8_t *x2;               // [n][kRes2Bytes]
    int8_t *tap[4], *tap_x2;  // outputs of the block convs and of the pool, or null
    int batch;
    Route route;
    int *status;
    uint64_t pad = 0;
    ResLayer layer[5];
};

struct ResStack23Params {  // two blocks at 20 x 20, conv, max-pool, two blocks at 9 x 9
    const int8_t *x2;
    const uint8_t *w;
    int8_t *x3;               // [n][kRes3Bytes], ReLU'd
    int8_t *tap[9], *tap_x3;  // outputs of the convs (not the last one) and of the pool, or null
    int batch;
    Route route;
    int *status;
    ResLayer layer[9];
};

// (By padding, not by a declared alignment: told of one, the compiler fetches by loads what are operands now, and with
// the layers in front of the other parameters some of the first kernel's; steps get 2 % slower, stacks 2 and 3 of
// 16384 images 710 us instead of 671.)
static_assert(sizeof(ResLayer) % 16 == 0 && offsetof(ResFirstParams, layer) % 16 == 0 && offsetof(ResStack1Params, layer) % 16 == 0 &&
              offsetof(ResStack23Params, layer) % 16 == 0, "16-byte reads");

cudaError_t res_first_launch(const ResFirstParams &p, int sm_count, cudaStream_t st);
cudaError_t res_stack1_launch(const ResStack1Params &p, int sm_count, cudaStream_t st);
cudaError_t res_stack23_launch(const ResStack23Params &p, int sm_count, cudaStream_t st);

}  // namespace accerl
