// One layer of the calibration pass (Section 2.2, "Parameter Quantization"): the int8 network so far is
// run layer by layer, and every layer twice -- first for the largest |epilogue value| of the batch, from
// which its output scale comes, then for its codes.  The contraction is cheap and its accumulators are not:
// written out as int32 they are four to sixteen times the layer's input (115 MB for the residual
// network's first layer and 256 frames).
//
// Warp-level int8 tensor instructions (m16n8k32) on NHWC words: a warp owns 32 output positions and up to
// 32 channels.  For one kernel row ky the window of a position is ONE run of consecutive words of the image
// row, so K is cut into pieces of eight words whatever the channel count; words outside the image are zeros.
// (The tcgen05 plans need operand layouts per shape and exist only once the scales do; this serves every
// shape the CUDA-core kernels serve.)  Sums are integers and the maximum is order-independent, so the scales
// and codes do not depend on the launch shape.  Bound by the loads of the operand words and, for small
// layers, by the launches.
#include "epilogue.cuh"
#include "internal.h"

namespace accerl {

namespace {

constexpr int kWarps = 4, kWarpRows = 32;      // of a block; positions of a warp (two 16-row tiles)
constexpr int kChunk = 64;                     // words of K whose weights are in shared memory at a time

struct CalibArgs {
    const int32_t *in;    // [n][H][W][C4] words
    const int32_t *skip;  // [position][out_cp / 4] words of the residual source, or null
    const int32_t *w;     // conv: [ky][run][oc_pad] words, fully connected: [oc_pad][run]
    const float *kscale, *bias;
    const int32_t *skip_mul;
    uint32_t *out;        // CODES: [position][out_cp / 4] words
    float *ymax;          // the largest |y|: written first, read for the codes
    long long total;      // output positions
    int H, W, C4, OH, OW, KH, run, stride, pad, oc_pad, out_cp;  // run: words of a window in one image row
    int relu_in, relu_out;
};

__device__ __forceinline__ void mma_s8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// NT: 8-column tiles of a block (16 or 32 output channels).  The columns are dealt out so that a thread's
// 2 * NT accumulators of a position are consecutive channels: column n of tile j is channel
// 2 * NT * (n / 2) + 2 * j + n % 2 of the block's.
template <int NT, bool FC, bool CODES>
__global__ void __launch_bounds__(32 * kWarps) calib_kernel(const CalibArgs a)
{
    constexpr int kStride = 8 * NT + 2;  // words of a row of weights (conflict-free for NT = 4)
    __shared__ int32_t s_w[kChunk * kStride];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int oc0 = blockIdx.y * 8 * NT;
    // this thread's four positions: rows g and g + 8 of two tiles
    long long px[4];
    const int32_t *row[4];  // first word of the position's window in image row iy0 (possibly outside the image)
    int iy0[4], x0[4];      // x0: that word's place in its image row
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        px[r] = ((long long)blockIdx.x * kWarps + warp) * kWarpRows + 8 * r + g;
        const long long q = px[r] < a.total ? px[r] : 0;
        const int ox = (int)(q % a.OW);
        const long long u = q / a.OW;
        const int oy = (int)(u % a.OH);
        iy0[r] = oy * a.stride - a.pad;
        x0[r] = (ox * a.stride - a.pad) * a.C4;
        row[r] = a.in + (u / a.OH * a.H + iy0[r]) * (long long)a.W * a.C4 + x0[r];
    }
    const int width = a.W * a.C4;
    int acc[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][j][i] = 0;
    for (int ky = 0; ky < a.KH; ++ky)
        for (int k0 = 0; k0 < a.run; k0 += kChunk) {
            const int words = min(kChunk, a.run - k0), padded = (words + 7) & ~7;
            __syncthreads();
            for (int i = threadIdx.x; i < padded * 8 * NT; i += 32 * kWarps) {
                const int k = FC ? i % padded : i / (8 * NT), c = FC ? i / padded : i % (8 * NT);
                int v = 0;
                if (k < words && oc0 + c < a.oc_pad)
                    v = FC ? __ldg(a.w + (size_t)(oc0 + c) * a.run + k0 + k) : __ldg(a.w + ((size_t)ky * a.run + k0 + k) * a.oc_pad + oc0 + c);
                s_w[k * kStride + c] = v;
            }
            __syncthreads();
            for (int k = 0; k < padded; k += 8) {
                uint32_t x[2][4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int at = k0 + k + 4 * h + t;
                        uint32_t v = 0;
                        if (at < a.run && (unsigned)(iy0[r] + ky) < (unsigned)a.H && (unsigned)(x0[r] + at) < (unsigned)width)
                            v = (uint32_t)__ldg(row[r] + (long long)ky * width + at);
                        x[r >> 1][(r & 1) + 2 * h] = a.relu_in ? relu_bytes(v) : v;
                    }
                const int32_t *w0 = s_w + (k + t) * kStride + 2 * NT * (g >> 1) + (g & 1), *w1 = w0 + 4 * kStride;
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const uint32_t b0 = (uint32_t)w0[2 * j], b1 = (uint32_t)w1[2 * j];
#pragma unroll
                    for (int m = 0; m < 2; ++m) mma_s8(acc[m][j], x[m], b0, b1);
                }
            }
        }
    // epilogue: 2 * NT channels from c0 on, of four positions
    const int c0 = oc0 + 2 * NT * t;
    float ymax = 0.f, s_out = 1.f;
    if (CODES) {
        const float m = *a.ymax;
        s_out = m > 0.f ? __fdiv_rn(m, 127.0f) : 1.0f;
    }
#pragma unroll
    for (int j = 0; j < NT; j += 2) {  // four channels at a time
        const int c = c0 + 2 * j;
        if (c >= a.out_cp) continue;
        const float4 k = *reinterpret_cast<const float4 *>(a.kscale + c), b = *reinterpret_cast<const float4 *>(a.bias + c);
        int4 mul = make_int4(0, 0, 0, 0);
        if (a.skip) mul = *reinterpret_cast<const int4 *>(a.skip_mul + c);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (px[r] >= a.total) continue;
            const int(&lo)[4] = acc[r >> 1][j], (&hi)[4] = acc[r >> 1][j + 1];
            int v[4] = {lo[2 * (r & 1)], lo[2 * (r & 1) + 1], hi[2 * (r & 1)], hi[2 * (r & 1) + 1]};
            const long long word = (px[r] * a.out_cp + c) / 4;
            if (a.skip) {
                const int sv = __ldg(a.skip + word);
                v[0] += mul.x * (int)(int8_t)sv;
                v[1] += mul.y * (int)(int8_t)(sv >> 8);
                v[2] += mul.z * (int)(int8_t)(sv >> 16);
                v[3] += mul.w * (int)(int8_t)(sv >> 24);
            }
            const float y[4] = {epilogue_float(v[0], k.x, b.x, a.relu_out), epilogue_float(v[1], k.y, b.y, a.relu_out),
                                epilogue_float(v[2], k.z, b.z, a.relu_out), epilogue_float(v[3], k.w, b.w, a.relu_out)};
            if (CODES)
                a.out[word] = (uint32_t)(uint8_t)requant(y[0], s_out) | (uint32_t)(uint8_t)requant(y[1], s_out) << 8 |
                              (uint32_t)(uint8_t)requant(y[2], s_out) << 16 | (uint32_t)(uint8_t)requant(y[3], s_out) << 24;
            else ymax = fmaxf(ymax, fmaxf(fmaxf(fabsf(y[0]), fabsf(y[1])), fmaxf(fabsf(y[2]), fabsf(y[3]))));
        }
    }
    if (!CODES) {  // (values >= 0: their bit patterns order like the values)
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(ymax));
        if (lane == 0 && m) atomicMax(reinterpret_cast<unsigned *>(a.ymax), m);
    }
}

template <int NT, bool FC>
void calib_go(const CalibArgs &a, cudaStream_t st)
{
    const dim3 grid((unsigned)((a.total + kWarps * kWarpRows - 1) / (kWarps * kWarpRows)), (unsigned)((a.oc_pad + 8 * NT - 1) / (8 * NT)));
    calib_kernel<NT, FC, false><<<grid, 32 * kWarps, 0, st>>>(a);
    calib_kernel<NT, FC, true><<<grid, 32 * kWarps, 0, st>>>(a);
}

}  // namespace

// B states: the largest |epilogue value| of layer L into *ymax (which must hold 0), its codes into `out`
cudaError_t launch_calib_layer(const LayerPlan &L, const int8_t *in, const int8_t *skip, int8_t *out, float *ymax, int B, cudaStream_t st)
{
    const bool fc = L.kind == ACCERL_FC;
    CalibArgs a;
    a.in = (const int32_t *)in;
    a.skip = (const int32_t *)skip;
    a.w = L.w_generic;
    a.kscale = L.kscale;
    a.bias = L.bias;
    a.skip_mul = L.skip_mul;
    a.out = (uint32_t *)out;
    a.ymax = ymax;
    a.oc_pad = L.oc_pad;
    a.out_cp = L.out_cp;
    a.relu_in = (L.flags & ACCERL_RELU_IN) != 0;
    a.relu_out = (L.flags & ACCERL_RELU_OUT) != 0;
    if (fc) {  // a window that is the whole row
        a.H = a.W = a.OH = a.OW = a.KH = a.stride = 1;
        a.pad = 0;
        a.C4 = a.run = L.in_cp * L.in_h * L.in_w / 4;
        a.total = B;
    } else {
        a.H = L.in_h; a.W = L.in_w; a.C4 = L.in_cp / 4; a.OH = L.out_h; a.OW = L.out_w;
        a.KH = L.kh; a.run = L.kw * a.C4; a.stride = L.stride; a.pad = L.pad;
        a.total = (long long)B * L.out_h * L.out_w;
    }
    if (L.oc_pad <= 16) fc ? calib_go<2, true>(a, st) : calib_go<2, false>(a, st);
    else fc ? calib_go<4, true>(a, st) : calib_go<4, false>(a, st);
    return cudaGetLastError();
}

}  // namespace accerl
