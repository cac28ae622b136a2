// Post-training quantisation on the device (Section 2.2, paragraphs "Parameter Quantization" and
// "Structured Pruning"): accerl_policy_create_fp32 takes the fp32 network the Learner trains and a
// calibration batch, and does what the Compressor's quantiser does before it hands the Actor a
// policy -- optional 2:4 pruning, symmetric int8 weights with one scale per output channel
// (max|w| / 127), one scale per activation tensor (max-abs of the epilogue float over the
// calibration batch, pushed through the already quantised preceding layers), the integer
// multipliers of the residual adds -- and then builds the handle with accerl_policy_create.
//
// The Compressor runs this for every policy it hands over, so it is a path of its own: one block of
// device memory, the contractions on the dp4a kernels (NHWC words) with the maximum of the epilogue
// value taken as they go, and no host round trip between the layers -- scales, epilogue constants and
// residual multipliers are computed where the maxima lie.  Every result is order-independent (integer
// sums, maxima), so the scales and codes are the same bits whatever the launch shape.  (One thread per
// output walking NCHW bytes, an atomic maximum per element and ten blocking copies a layer took 44 ms
// for the residual network with 256 calibration frames, building the handle included; now 9.)  The
// Actor step itself never runs these kernels.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "epilogue.cuh"
#include "internal.h"

namespace accerl {

namespace {

// the scale max-abs calibration gives (1 where nothing was seen)
__device__ __forceinline__ float scale_of(float ymax) { return ymax > 0.f ? __fdiv_rn(ymax, 127.0f) : 1.0f; }

__device__ __forceinline__ void warp_max_to(float v, float *out)  // v >= 0: the bit patterns order like the values
{
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(reinterpret_cast<unsigned *>(out), m);
}

// 2:4 pruning along K = (kh, kw, c_in), c_in fastest: of every four consecutive K positions keep
// the two of largest |w| (the lower index wins a tie), zero the others.  In place, OIHW.
__global__ void prune24_kernel(float *w, int oc, int ic, int kh, int kw)
{
    const long long groups = (long long)oc * kh * kw * ic / 4;
    const long long gidx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gidx >= groups) return;
    const int per_oc = kh * kw * ic / 4;
    const int o = (int)(gidx / per_oc);
    const int k0 = (int)(gidx - (long long)o * per_oc) * 4;
    float v[4];
    long long at[4];
    for (int j = 0; j < 4; ++j) {
        const int k = k0 + j, c = k % ic, t = k / ic, x = t % kw, y = t / kw;
        at[j] = (((long long)o * ic + c) * kh + y) * kw + x;
        v[j] = w[at[j]];
    }
    // rank of element j: how many others come before it in a stable sort by decreasing |w|
    for (int j = 0; j < 4; ++j) {
        int before = 0;
        for (int i = 0; i < 4; ++i)
            if (i != j && (fabsf(v[i]) > fabsf(v[j]) || (fabsf(v[i]) == fabsf(v[j]) && i < j))) ++before;
        if (before >= 2) w[at[j]] = 0.f;
    }
}

// one block per output channel: s_w = max|w| / 127 (1 for an all-zero row), q = clip(rint(w / s_w))
__global__ void quantise_weights_kernel(const float *w, int K, float *s_w, int8_t *q)
{
    __shared__ float red[256];
    const int o = blockIdx.x;
    const float *row = w + (long long)o * K;
    float m = 0.f;
    for (int k = threadIdx.x; k < K; k += blockDim.x) m = fmaxf(m, fabsf(row[k]));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    const float s = red[0] > 0.f ? __fdiv_rn(red[0], 127.0f) : 1.0f;
    if (threadIdx.x == 0) s_w[o] = s;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        float t = rintf(__fdiv_rn(row[k], s));
        t = fminf(fmaxf(t, -127.f), 127.f);
        q[(long long)o * K + k] = (int8_t)t;
    }
}

// max |x| of the real-valued input: frames are u / 255 (non-decreasing in u), vectors are taken as they are
__global__ void input_absmax_u8_kernel(const uint8_t *obs, long long n, float *out)
{
    const long long words = n / 16, first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
    unsigned m = 0;
    for (long long i = first; i < words; i += stride) {
        const uint4 v = reinterpret_cast<const uint4 *>(obs)[i];
        m = __vmaxu4(m, __vmaxu4(__vmaxu4(v.x, v.y), __vmaxu4(v.z, v.w)));
    }
    for (long long i = 16 * words + first; i < n; i += stride) m = __vmaxu4(m, obs[i]);
    const unsigned u = max(max(m & 0xff, (m >> 8) & 0xff), max((m >> 16) & 0xff, m >> 24));
    warp_max_to(__fdiv_rn((float)u, 255.0f), out);
}

__global__ void input_absmax_f32_kernel(const float *obs, long long n, float *out)
{
    float m = 0.f;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(obs[i]));
    warp_max_to(m, out);
}

__device__ __forceinline__ int8_t quantise_real(float x, float s) { return (int8_t)clamp_round_i8(__fdiv_rn(x, s)); }

// the 256-entry input table of launch_ingest_u8
__global__ void input_table_kernel(const float *ymax, int8_t *lut)
{
    lut[threadIdx.x] = quantise_real(__fdiv_rn((float)threadIdx.x, 255.0f), scale_of(*ymax));
}

__global__ void input_quantise_f32_kernel(const float *obs, long long rows, int D, int pitch, const float *ymax, int8_t *q)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * pitch) return;
    const long long r = i / pitch;
    const int k = (int)(i - r * pitch);
    q[i] = k < D ? quantise_real(obs[r * D + k], scale_of(*ymax)) : 0;
}

// int8 OIHW weights -> the word layouts of the dp4a kernels (see pack_generic): one byte per thread
__global__ void pack_conv_kernel(const int8_t *w, long long n, int ic, int taps, int oc_pad, int8_t *out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int tap = (int)(i % taps), c = (int)(i / taps % ic), o = (int)(i / taps / ic), c4 = (ic + 3) / 4;
    out[(((size_t)tap * c4 + c / 4) * oc_pad + o) * 4 + c % 4] = w[i];
}
__global__ void pack_fc_kernel(const int8_t *w, long long n, int C, int HW, int pitch, int8_t *out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int hw = (int)(i % HW), c = (int)(i / HW % C);
    const long long o = i / HW / C;
    out[o * (long long)HW * pitch + (size_t)hw * pitch + c] = w[i];
}

// epilogue constants of a layer: k = s_in * s_w, rounded once, and the integer multiplier that brings
// the skip tensor (scale s_x) onto the accumulators' grid
__global__ void layer_scales_kernel(const float *s_w, int oc, const float *ymax_in, const float *ymax_skip, float *k, int *mul)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= oc) return;
    const float kc = __fmul_rn(scale_of(*ymax_in), s_w[c]);
    k[c] = kc;
    if (ymax_skip) mul[c] = (int)fminf(fmaxf(rintf(__fdiv_rn(scale_of(*ymax_skip), kc)), 0.f), 32767.f);
}

// accumulators -> codes, four channels per thread
__global__ void calib_requant_kernel(const int4 *acc, const float *k, const float *b, int relu, int c4s, long long words,
                                     const float *ymax, uint32_t *q)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    const int c = (int)(i % c4s) * 4;
    const int4 a = acc[i];
    const float s = scale_of(*ymax);
    q[i] = (uint32_t)(uint8_t)requant(epilogue_float(a.x, k[c], b[c], relu), s) |
           (uint32_t)(uint8_t)requant(epilogue_float(a.y, k[c + 1], b[c + 1], relu), s) << 8 |
           (uint32_t)(uint8_t)requant(epilogue_float(a.z, k[c + 2], b[c + 2], relu), s) << 16 |
           (uint32_t)(uint8_t)requant(epilogue_float(a.w, k[c + 3], b[c + 3], relu), s) << 24;
}

// one block of device memory, handed out piece by piece: sized in a first pass, filled in a second
struct DeviceArena {
    char *base = nullptr;
    size_t at = 0;
    ~DeviceArena()
    {
        // (where a call failed, its kernels may still run)
        if (base) device_free(base, cudaStreamSynchronize(0) == cudaSuccess);
    }
    template <typename T>
    T *take(size_t count)
    {
        T *p = (T *)(base + at);  // (meaningless while base is null: the sizing pass)
        at += (count * sizeof(T) + 255) / 256 * 256;
        return p;
    }
};

unsigned blocks_for(long long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

}  // namespace accerl

using namespace accerl;

static accerl_status quantise_and_create(accerl_policy **out, int32_t in_kind,
                                                   const int32_t in_shape[3],
                                                   const accerl_layer_fp32 *layers, int32_t n_layers,
                                                   const void *calib_obs_host, int32_t calib_rows,
                                                   int32_t prune_2_4, int32_t max_batch, uint32_t flags,
                                                   int32_t device)
{
    if (out) *out = nullptr;
    if (!out || !in_shape || !layers || !calib_obs_host) {
        set_error("create_fp32: null argument");
        return ACCERL_ERR_INVALID_ARG;
    }
    if ((in_kind != ACCERL_IN_U8_NCHW && in_kind != ACCERL_IN_F32) || n_layers < 1 || n_layers > 4096 ||
        calib_rows < 1 || calib_rows > (1 << 20) || in_shape[0] < 1 || in_shape[1] < 1 || in_shape[2] < 1) {
        set_error("create_fp32: bad input kind, shape, layer count or calibration rows");
        return ACCERL_ERR_INVALID_ARG;
    }
    // shapes (the full validation is accerl_policy_create's; here only what the kernels index with)
    struct Shape {
        int c, h, w;
    };
    std::vector<Shape> shapes;
    Shape cur{in_shape[0], in_shape[1], in_shape[2]};
    size_t max_elems = (size_t)cur.c * cur.h * cur.w;
    for (int i = 0; i < n_layers; ++i) {
        const accerl_layer_fp32 &d = layers[i];
        Shape o;
        if (d.kind == ACCERL_FC) {
            if ((long long)cur.c * cur.h * cur.w != d.in_c || d.out_c < 1) {
                set_error("create_fp32: layer %d: FC expects in_c = %lld", i, (long long)cur.c * cur.h * cur.w);
                return ACCERL_ERR_INVALID_ARG;
            }
            o = Shape{d.out_c, 1, 1};
        } else if (d.kind == ACCERL_CONV2D || d.kind == ACCERL_MAXPOOL) {
            if (d.in_c != cur.c || d.in_h != cur.h || d.in_w != cur.w || d.kh < 1 || d.kw != d.kh || d.stride < 1 ||
                d.pad < 0 || d.pad >= d.kh || d.out_c < 1 || cur.h + 2 * d.pad < d.kh || cur.w + 2 * d.pad < d.kw ||
                (d.kind == ACCERL_MAXPOOL && (d.pad != 0 || d.out_c != d.in_c))) {
                set_error("create_fp32: layer %d: shape does not follow from the previous layer", i);
                return ACCERL_ERR_INVALID_ARG;
            }
            o = Shape{d.out_c, (cur.h + 2 * d.pad - d.kh) / d.stride + 1, (cur.w + 2 * d.pad - d.kw) / d.stride + 1};
        } else {
            set_error("create_fp32: layer %d: unknown kind %d", i, d.kind);
            return ACCERL_ERR_INVALID_ARG;
        }
        if (d.kind != ACCERL_MAXPOOL && (!d.w || !d.bias)) {
            set_error("create_fp32: layer %d: w and bias must be non-null", i);
            return ACCERL_ERR_INVALID_ARG;
        }
        if (d.skip_from >= i || d.skip_from < -1 ||
            (d.skip_from >= 0 && (d.kind != ACCERL_CONV2D || shapes[d.skip_from].c != o.c ||
                                  shapes[d.skip_from].h != o.h || shapes[d.skip_from].w != o.w))) {
            set_error("create_fp32: layer %d: skip_from must name an earlier layer with this layer's output shape", i);
            return ACCERL_ERR_INVALID_ARG;
        }
        if (prune_2_4 && d.kind != ACCERL_MAXPOOL && ((long long)d.in_c * d.kh * d.kw) % 4) {
            set_error("create_fp32: layer %d: 2:4 pruning needs K to be a multiple of 4", i);
            return ACCERL_ERR_INVALID_ARG;
        }
        shapes.push_back(o);
        max_elems = std::max(max_elems, (size_t)o.c * o.h * o.w);
        cur = o;
    }
    if (max_elems * (size_t)calib_rows >= ((size_t)1 << 33)) {
        set_error("create_fp32: calibration batch too large (%zu elements per tensor)", max_elems * (size_t)calib_rows);
        return ACCERL_ERR_UNSUPPORTED;
    }
    int ndev = 0, prev = -1;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        set_error("create_fp32: CUDA device %d not available", device);
        cudaGetLastError();
        return ACCERL_ERR_CUDA;
    }
    cudaGetDevice(&prev);
    struct Restore {
        int prev;
        ~Restore() { if (prev >= 0) cudaSetDevice(prev); }
    } restore{prev};
    ACCERL_CUDA_TRY(cudaSetDevice(device));

    const long long B = calib_rows;
    const long long in_elems = (long long)in_shape[0] * in_shape[1] * in_shape[2] * B;
    const bool u8 = in_kind == ACCERL_IN_U8_NCHW;
    struct Layer {
        LayerPlan L;      // the dp4a kernels' view of the layer
        int8_t *act;      // its int8 output, NHWC
        float *w;
        int8_t *wq, *packed;
        float *s_w, *k, *b;
        int *mul;
        size_t nw, packed_bytes;
        int scale;        // index of the maximum its output scale comes from (a pool passes its input's on)
    };
    std::vector<Layer> net(n_layers);
    int n_run = n_layers;  // layers up to the one with the logits
    DeviceArena mem;
    void *obs_dev = nullptr;
    int8_t *lut = nullptr, *act0 = nullptr;
    float *ymax = nullptr;
    int *acc = nullptr;
    char *results = nullptr;  // what goes back to the host, in one piece: wq, s_w and mul of every layer, ymax
    size_t results_bytes = 0;
    for (int pass = 0; pass < 2; ++pass) {
        mem.at = 0;
        results = mem.take<char>(0);
        ymax = mem.take<float>(n_layers + 1);
        Shape in{in_shape[0], in_shape[1], in_shape[2]};
        for (int i = 0; i < n_layers; ++i) {
            const accerl_layer_fp32 &d = layers[i];
            Layer &l = net[i];
            LayerPlan &L = l.L;
            L.kind = d.kind;
            L.flags = d.flags;
            L.in_c = in.c; L.in_h = in.h; L.in_w = in.w; L.in_cp = round_up(in.c, 4);
            L.out_c = shapes[i].c; L.out_h = shapes[i].h; L.out_w = shapes[i].w; L.out_cp = round_up(shapes[i].c, 4);
            L.oc_pad = round_up(L.out_c, 16);
            L.kh = d.kh; L.kw = d.kw; L.stride = d.stride; L.pad = d.pad;
            L.skip_from = d.skip_from;
            l.nw = l.packed_bytes = 0;
            if (d.kind != ACCERL_MAXPOOL) {
                const int taps = d.kind == ACCERL_FC ? 1 : d.kh * d.kw;
                l.nw = (size_t)d.out_c * (d.kind == ACCERL_FC ? d.in_c : in.c * taps);
                l.packed_bytes = d.kind == ACCERL_FC ? (size_t)L.oc_pad * in.h * in.w * L.in_cp : (size_t)taps * L.in_cp * L.oc_pad;
            }
            l.wq = mem.take<int8_t>(l.nw);
            l.s_w = mem.take<float>(l.nw ? d.out_c : 0);
            l.mul = mem.take<int>(d.skip_from >= 0 ? L.oc_pad : 0);
            in = shapes[i];
            if ((d.flags & ACCERL_LOGITS) && n_run > i + 1) n_run = i + 1;
        }
        results_bytes = mem.at;
        // (from here on nothing has to start at zero but the packed weights and the padded constants)
        const size_t zero_from = mem.at;
        for (int i = 0; i < n_layers; ++i) {
            Layer &l = net[i];
            l.packed = mem.take<int8_t>(l.packed_bytes);
            l.k = mem.take<float>(l.nw ? l.L.oc_pad : 0);
            l.b = mem.take<float>(l.nw ? l.L.oc_pad : 0);
        }
        const size_t zero_to = mem.at;
        for (int i = 0; i < n_layers; ++i) net[i].w = mem.take<float>(net[i].nw);
        obs_dev = mem.take<uint8_t>((size_t)in_elems * (u8 ? 1 : 4));
        lut = mem.take<int8_t>(256);
        act0 = mem.take<int8_t>((size_t)B * in_shape[1] * in_shape[2] * round_up(in_shape[0], 4));
        size_t acc_elems = 0;
        for (int i = 0; i < n_layers; ++i) {
            const LayerPlan &L = net[i].L;
            const size_t elems = (size_t)B * L.out_h * L.out_w * L.out_cp;
            net[i].act = mem.take<int8_t>(elems);
            if (net[i].nw) acc_elems = std::max(acc_elems, elems);
        }
        acc = mem.take<int>(acc_elems);
        if (pass == 0) {
            ACCERL_CUDA_TRY(device_alloc((void **)&mem.base, mem.at + 256));
            continue;
        }
        ACCERL_CUDA_TRY(cudaMemsetAsync(ymax, 0, (n_layers + 1) * sizeof(float), 0));
        for (int i = 0; i < n_layers; ++i)
            if (layers[i].skip_from >= 0) ACCERL_CUDA_TRY(cudaMemsetAsync(net[i].mul, 0, net[i].L.oc_pad * sizeof(int), 0));
        ACCERL_CUDA_TRY(cudaMemsetAsync(mem.base + zero_from, 0, zero_to - zero_from, 0));
    }

    // ---- the calibration batch, quantised (ymax[0]: its maximum), and the weights
    ACCERL_CUDA_TRY(cudaMemcpyAsync(obs_dev, calib_obs_host, (size_t)in_elems * (u8 ? 1 : 4), cudaMemcpyHostToDevice, 0));
    if (u8) {
        input_absmax_u8_kernel<<<592, 256>>>((const uint8_t *)obs_dev, in_elems, ymax);
        input_table_kernel<<<1, 256>>>(ymax, lut);
        ACCERL_CUDA_TRY(launch_ingest_u8((const uint8_t *)obs_dev, lut, act0, (int)B, in_shape[0], in_shape[1], in_shape[2],
                                         round_up(in_shape[0], 4), 0));
    } else {
        const int pitch = round_up(in_shape[0], 4);
        input_absmax_f32_kernel<<<592, 256>>>((const float *)obs_dev, in_elems, ymax);
        input_quantise_f32_kernel<<<blocks_for(B * pitch), 256>>>((const float *)obs_dev, B, in_shape[0], pitch, ymax, act0);
    }
    ACCERL_CUDA_TRY(cudaGetLastError());
    for (int i = 0; i < n_layers; ++i) {
        const accerl_layer_fp32 &d = layers[i];
        Layer &l = net[i];
        if (!l.nw) continue;
        ACCERL_CUDA_TRY(cudaMemcpyAsync(l.w, d.w, l.nw * 4, cudaMemcpyHostToDevice, 0));
        ACCERL_CUDA_TRY(cudaMemcpyAsync(l.b, d.bias, (size_t)d.out_c * 4, cudaMemcpyHostToDevice, 0));
        const int ic = d.in_c, kh = d.kind == ACCERL_FC ? 1 : d.kh;
        if (prune_2_4) prune24_kernel<<<blocks_for((long long)l.nw / 4), 256>>>(l.w, d.out_c, ic, kh, kh);
        quantise_weights_kernel<<<(unsigned)d.out_c, 256>>>(l.w, (int)(l.nw / d.out_c), l.s_w, l.wq);
        if (d.kind == ACCERL_FC)
            pack_fc_kernel<<<blocks_for((long long)l.nw), 256>>>(l.wq, (long long)l.nw, l.L.in_c, l.L.in_h * l.L.in_w, l.L.in_cp, l.packed);
        else
            pack_conv_kernel<<<blocks_for((long long)l.nw), 256>>>(l.wq, (long long)l.nw, d.in_c, kh * kh, l.L.oc_pad, l.packed);
        ACCERL_CUDA_TRY(cudaGetLastError());
        l.L.w_generic = (int32_t *)l.packed;
        l.L.kscale = l.k;
        l.L.bias = l.b;
        l.L.skip_mul = d.skip_from >= 0 ? l.mul : nullptr;
    }

    // ---- layer by layer
    int s_in = 0;  // index of the input scale's maximum
    for (int i = 0; i < n_run; ++i) {
        const accerl_layer_fp32 &d = layers[i];
        Layer &l = net[i];
        const int8_t *x = i ? net[i - 1].act : act0;
        l.scale = i + 1;
        if (d.kind == ACCERL_MAXPOOL) {
            l.scale = s_in;
            ACCERL_CUDA_TRY(launch_maxpool_generic(l.L, x, l.act, (int)B, 0));
            continue;
        }
        layer_scales_kernel<<<(unsigned)((d.out_c + 127) / 128), 128>>>(l.s_w, d.out_c, ymax + s_in,
                                                                        d.skip_from >= 0 ? ymax + net[d.skip_from].scale : nullptr, l.k, l.mul);
        ACCERL_CUDA_TRY(cudaGetLastError());
        if (d.flags & ACCERL_LOGITS) break;  // its output is not quantised
        if (d.kind == ACCERL_FC) ACCERL_CUDA_TRY(launch_fc_acc(l.L, x, acc, ymax + i + 1, (int)B, 0));
        else
            ACCERL_CUDA_TRY(launch_conv_acc(l.L, x, d.skip_from >= 0 ? net[d.skip_from].act : nullptr, acc, ymax + i + 1, (int)B, 0));
        const long long words = B * l.L.out_h * l.L.out_w * (l.L.out_cp / 4);
        calib_requant_kernel<<<blocks_for(words), 256>>>((const int4 *)acc, l.k, l.b, (d.flags & ACCERL_RELU_OUT) ? 1 : 0,
                                                         l.L.out_cp / 4, words, ymax + i + 1, (uint32_t *)l.act);
        ACCERL_CUDA_TRY(cudaGetLastError());
        s_in = i + 1;
    }
    // one block, kept as it comes back: copies of its parts cost their page faults again
    std::shared_ptr<char[]> back;
    std::vector<accerl_policy::PtqLayer> Q(n_layers);
    ACCERL_CUDA_TRY(pinned_alloc(&back, results_bytes));
    ACCERL_CUDA_TRY(cudaMemcpy(back.get(), results, results_bytes, cudaMemcpyDeviceToHost));
    auto host = [&](const void *dev) { return back.get() + ((const char *)dev - results); };
    auto scale = [&](int at) {
        const float m = reinterpret_cast<const float *>(host(ymax))[at];
        volatile float s = m > 0.f ? m / 127.0f : 1.0f;
        return (float)s;
    };
    const float s_input = scale(0);
    float s_prev = s_input;
    for (int i = 0; i < n_run; ++i) {
        const accerl_layer_fp32 &d = layers[i];
        const Layer &l = net[i];
        accerl_policy::PtqLayer &q = Q[i];
        q.s_in = s_prev;
        q.s_out = (d.flags & ACCERL_LOGITS) ? 1.0f : scale(l.scale);
        s_prev = q.s_out;
        if (!l.nw) continue;
        q.w = (const int8_t *)host(l.wq);
        q.n_w = l.nw;
        q.s_w = (const float *)host(l.s_w);
        q.n_s_w = (size_t)d.out_c;
        if (d.skip_from >= 0) {
            q.skip_mul = (const int32_t *)host(l.mul);
            q.n_skip_mul = (size_t)d.out_c;
        }
    }

    // ---- hand the quantised network to the ordinary constructor
    std::vector<accerl_layer_desc> descs(n_layers);
    for (int i = 0; i < n_layers; ++i) {
        const accerl_layer_fp32 &d = layers[i];
        accerl_layer_desc &e = descs[i];
        memset(&e, 0, sizeof(e));
        e.kind = d.kind;
        e.flags = d.flags;
        e.in_c = d.in_c; e.in_h = d.in_h; e.in_w = d.in_w; e.out_c = d.out_c;
        e.kh = d.kh; e.kw = d.kw; e.stride = d.stride; e.pad = d.pad;
        e.s_in = Q[i].s_in;
        e.s_out = Q[i].s_out;
        e.skip_from = d.skip_from;
        if (d.kind != ACCERL_MAXPOOL) {
            e.w = Q[i].w;
            e.s_w = Q[i].s_w;
            e.bias = d.bias;
            e.skip_mul = Q[i].skip_mul;
        }
    }
    accerl_status st = accerl_policy_create(out, in_kind, in_shape, s_input, descs.data(), n_layers, max_batch,
                                            flags, device);
    if (st != ACCERL_OK) return st;
    // keep the quantised parameters for accerl_policy_export
    accerl_policy *p = *out;
    p->ptq = std::move(Q);
    p->ptq_data = std::move(back);
    return ACCERL_OK;
}

extern "C" accerl_status accerl_policy_create_fp32(accerl_policy **out, int32_t in_kind,
                                                   const int32_t in_shape[3],
                                                   const accerl_layer_fp32 *layers, int32_t n_layers,
                                                   const void *calib_obs_host, int32_t calib_rows,
                                                   int32_t prune_2_4, int32_t max_batch, uint32_t flags,
                                                   int32_t device)
{
    try {
        return quantise_and_create(out, in_kind, in_shape, layers, n_layers, calib_obs_host, calib_rows, prune_2_4, max_batch, flags,
                                   device);
    } catch (const std::bad_alloc &) {
        set_error("create_fp32: out of host memory");
        return ACCERL_ERR_OOM;
    }
}

extern "C" accerl_status accerl_policy_export(const accerl_policy *p, int32_t layer, int8_t *w_host,
                                              size_t w_bytes, float *s_w_host, int32_t *skip_mul_host,
                                              float *s_in_out, float *s_out_out)
{
    if (!p) {
        set_error("export: null handle");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (p->ptq.empty()) {
        set_error("export: the handle was not built by accerl_policy_create_fp32");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (layer < 0 || layer >= (int)p->ptq.size()) {
        set_error("export: layer %d out of range", layer);
        return ACCERL_ERR_INVALID_ARG;
    }
    const accerl_policy::PtqLayer &q = p->ptq[layer];
    if (s_in_out) *s_in_out = q.s_in;
    if (s_out_out) *s_out_out = q.s_out;
    if (w_host) {
        if (w_bytes < q.n_w) {
            set_error("export: w_host holds %zu bytes, %zu needed", w_bytes, q.n_w);
            return ACCERL_ERR_INVALID_ARG;
        }
        if (q.n_w) memcpy(w_host, q.w, q.n_w);
    }
    if (s_w_host && q.n_s_w) memcpy(s_w_host, q.s_w, q.n_s_w * sizeof(float));
    if (skip_mul_host && q.n_skip_mul) memcpy(skip_mul_host, q.skip_mul, q.n_skip_mul * sizeof(int32_t));
    return ACCERL_OK;
}
