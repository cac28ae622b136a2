// Small-batch latency path for all-FC policies on vector observations (the CartPole / LunarLander
// shaped networks at the paper's batch of 160 and up): the whole step -- input quantisation,
// every layer with its requantising epilogue, log-softmax, inverse-CDF sampling -- is ONE launch.
// At these sizes the step is bound by launch latency, not by arithmetic, so a chain of per-layer
// kernels would spend most of its time between kernels.
//
// A CTA owns 16 or 32 states.  Activations stay in shared memory as int8 rows; the layers run on
// warp-level int8 tensor instructions (m16n8k32), whose 16-row granule fits a handful of states per
// CTA -- a 128-row tile of the big tensor pipe would leave all but 32 SMs idle at 4096 states.  The
// sixteen warps share a layer's columns.  Weights and scales arrive by bulk copies (all layers at once
// where they fit, else two layers ahead), started before the previous launch has finished, and lie in
// the order the instruction's lanes want them: one conflict-free 8-byte load per instruction.
//
// What bounds it: every warp is one chain of dependent instructions, layer after layer, at eight-odd
// cycles each, so what counts is how many a warp has to run.  The dp4a form of this kernel (8 states
// per CTA, every weight word loaded from L2 by the thread that used it) took 21.8 us for 4096 states
// of 8-256-256-4; with the weights in registers, unrolled for the widest layer, 12 us; this form 8.2 us.
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "epilogue.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace accerl {

namespace {
constexpr int kMaxWidth = 256; // widest layer
constexpr int kMaxLayers = 8;
constexpr int kMlpWarps = 16;
constexpr int kMlpPitch = kMaxWidth / 4 + 4;  // words of an activation row: 4 mod 8, so that the eight rows and
                                              // four words of an operand load fall into 32 different banks
}  // namespace

struct MlpFusedParams {
    int n_layers, in_dim, n_actions;
    float s_input;
    int kt[kMaxLayers];        // 32-byte K steps of layer l
    int nt[kMaxLayers];        // 8-column tiles of layer l (a multiple of 4 except in the last)
    int n[kMaxLayers];         // outputs of layer l
    int relu[kMaxLayers];
    float s_out[kMaxLayers], inv_s_out[kMaxLayers];
    // layer l's block of parameters: [nt][kt][lane] 8-byte B operands, then 8 * nt scales and 8 * nt
    // biases (0 in padding columns)
    const uint8_t *block[kMaxLayers];
    uint32_t block_bytes[kMaxLayers];
    uint32_t slot_off[kMaxLayers];  // where it goes in shared memory
    int slots;                      // layers in flight: n_layers (every layer has its own place) or 2
    uint32_t smem_bytes;
    int *status;
    // parity taps (null without them): the quantised input and every hidden layer's int8 output
    // are also stored, rows of tap_in_pitch / tap_pitch[l] bytes
    int8_t *tap_in, *tap[kMaxLayers];
    int tap_in_pitch, tap_pitch[kMaxLayers];
};

__device__ __forceinline__ void mma_m16n8k32_s8(int (&d)[4], const uint32_t (&a)[4], uint2 b)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// the codes of one thread's four accumulators by the IEEE divide (out of line: rarely taken)
__device__ __noinline__ uint32_t exact_codes4(int a0, int a1, int a2, int a3, float2 ks, float2 bs, float s_out)
{
    return pack4_sat_s8(__float2int_rn(__fdiv_rn(epilogue_float(a0, ks.x, bs.x, false), s_out)),
                        __float2int_rn(__fdiv_rn(epilogue_float(a1, ks.y, bs.y, false), s_out)),
                        __float2int_rn(__fdiv_rn(epilogue_float(a2, ks.x, bs.x, false), s_out)),
                        __float2int_rn(__fdiv_rn(epilogue_float(a3, ks.y, bs.y, false), s_out)));
}

// MT: 16-row tiles of a CTA
template <int MT>
__global__ void __launch_bounds__(32 * kMlpWarps, 2)
mlp_fused_kernel(const __grid_constant__ MlpFusedParams p, const float *__restrict__ obs, const float *__restrict__ u,
                 int B, float *__restrict__ logits, int32_t *__restrict__ actions,
                 float *__restrict__ logp, float *__restrict__ value, float *__restrict__ entropy)
{
    constexpr int kRows = 16 * MT;
    extern __shared__ __align__(16) uint8_t mlp_smem[];
    __shared__ __align__(16) uint32_t act[2][kRows][kMlpPitch];
    __shared__ float s_logits[kRows][33];
    __shared__ __align__(8) uint64_t full[kMaxLayers];
    __shared__ int abort_flag;
    const int tid = threadIdx.x, row0 = blockIdx.x * kRows, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, q = lane & 3;  // the instruction's row group and column pair of a lane

    auto fetch = [&](int l) {  // one thread: layer l's parameters into its slot
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(smem_u32(&full[l]), p.block_bytes[l]);
        bulk_load(smem_u32(mlp_smem) + p.slot_off[l], p.block[l], p.block_bytes[l], smem_u32(&full[l]));
    };
    if (tid == 0) {
        for (int l = 0; l < p.n_layers; ++l) mbar_init(smem_u32(&full[l]), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int l = 0; l < p.slots; ++l) fetch(l);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // input quantisation into act[0], zero up to the next K step
    const int words0 = 8 * p.kt[0];
    for (int i = tid; i < kRows * words0; i += 32 * kMlpWarps) {
        const int r = i / words0, w4 = i - r * words0, row = row0 + r;
        uint32_t word = 0;
        if (row < B && 4 * w4 < p.in_dim) {
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                x[j] = 4 * w4 + j < p.in_dim ? __ldg(obs + (long long)row * p.in_dim + 4 * w4 + j) : 0.f;
#pragma unroll 1
            for (int j = 0; j < 4; ++j) {  // rolled: the divide is long
                word = (word >> 8) | (uint32_t)(uint8_t)quantise_input(x[0], p.s_input) << 24;
                x[0] = x[1];
                x[1] = x[2];
                x[2] = x[3];
            }
            if (p.tap_in && 4 * w4 < p.tap_in_pitch)
                *reinterpret_cast<uint32_t *>(p.tap_in + (long long)row * p.tap_in_pitch + 4 * w4) = word;
        }
        act[0][r][w4] = word;
    }
    __syncthreads();

    int cur = 0;
    for (int l = 0; l < p.n_layers; ++l) {
        const int KT = p.kt[l], NT = p.nt[l], N = p.n[l];
        const bool last = l == p.n_layers - 1;
        const uint8_t *blk = mlp_smem + p.slot_off[l];
        const float *s_ks = reinterpret_cast<const float *>(blk + NT * KT * 256), *s_bs = s_ks + 8 * NT;
        const float s_out = p.s_out[l], inv = p.inv_s_out[l];
        const bool relu = p.relu[l] != 0;
        if (warp < NT && !mbar_wait(smem_u32(&full[l]), 0, (volatile int *)&abort_flag, p.status, 1)) break;
        for (int nt = warp; nt < NT; nt += kMlpWarps) {
            int acc[MT][4] = {};
            const uint2 *wb = reinterpret_cast<const uint2 *>(blk) + nt * KT * 32 + lane;
            const uint32_t *xa = &act[cur][g][q];
#pragma unroll 2
            for (int k = 0; k < KT; ++k) {
                const uint2 w = wb[32 * k];
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const uint32_t *x = xa + 16 * m * kMlpPitch + 8 * k;
                    const uint32_t a[4] = {x[0], x[8 * kMlpPitch], x[4], x[8 * kMlpPitch + 4]};
                    mma_m16n8k32_s8(acc[m], a, w);
                }
            }
            const int col = 8 * nt + 2 * q;
            const float2 ks = *reinterpret_cast<const float2 *>(s_ks + col), bs = *reinterpret_cast<const float2 *>(s_bs + col);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float2 y0 = __ffma2_rn(make_float2(__int2float_rn(acc[m][0]), __int2float_rn(acc[m][1])), ks, bs);
                const float2 y1 = __ffma2_rn(make_float2(__int2float_rn(acc[m][2]), __int2float_rn(acc[m][3])), ks, bs);
                if (last) {  // (no ReLU on logits)
                    float *z0 = &s_logits[16 * m + g][col], *z1 = &s_logits[16 * m + g + 8][col];
                    if (col < N) z0[0] = relu ? fmaxf(y0.x, 0.f) : y0.x, z1[0] = relu ? fmaxf(y1.x, 0.f) : y1.x;
                    if (col + 1 < N) z0[1] = relu ? fmaxf(y0.y, 0.f) : y0.y, z1[1] = relu ? fmaxf(y1.y, 0.f) : y1.y;
                    continue;
                }
                // reciprocal first, the IEEE divide where that could round differently (see epilogue.cuh);
                // |t - rint(t)| by adding and subtracting 1.5 * 2^23 (for a |t| too large for that the
                // difference is garbage: at worst the divide is done for nothing).  ReLU is applied to the
                // codes, which have the sign of y.
                const float2 inv2 = make_float2(inv, inv), up2 = make_float2(kRoundMagic, kRoundMagic),
                             down2 = make_float2(-kRoundMagic, -kRoundMagic), neg2 = make_float2(-1.f, -1.f);
                const float2 t0 = __fmul2_rn(y0, inv2), t1 = __fmul2_rn(y1, inv2);
                const float2 d0 = __ffma2_rn(__fadd2_rn(__fadd2_rn(t0, up2), down2), neg2, t0);
                const float2 d1 = __ffma2_rn(__fadd2_rn(__fadd2_rn(t1, up2), down2), neg2, t1);
                const float worst = fmaxf(fmaxf(fabsf(d0.x), fabsf(d0.y)), fmaxf(fabsf(d1.x), fabsf(d1.y)));
                uint32_t packed = pack4_sat_s8(__float2int_rn(t0.x), __float2int_rn(t0.y), __float2int_rn(t1.x),
                                               __float2int_rn(t1.y));
                if (worst > 0.5f - kTieGuard)
                    packed = exact_codes4(acc[m][0], acc[m][1], acc[m][2], acc[m][3], ks, bs, s_out);
                if (relu) packed = relu_bytes(packed);
                uint8_t *dst = reinterpret_cast<uint8_t *>(act[cur ^ 1][16 * m + g]) + col;
                *reinterpret_cast<uint16_t *>(dst) = (uint16_t)packed;
                *reinterpret_cast<uint16_t *>(dst + 8 * 4 * kMlpPitch) = (uint16_t)(packed >> 16);
                if (p.tap[l]) {
#pragma unroll 1
                    for (int j = 0; j < 4; ++j) {
                        const int row = row0 + 16 * m + g + 8 * (j >> 1);
                        if (row < B && col + (j & 1) < N)
                            p.tap[l][(long long)row * p.tap_pitch[l] + col + (j & 1)] = (int8_t)(packed >> (8 * j));
                    }
                }
            }
        }
        __syncthreads();
        if (tid == 0 && l + p.slots < p.n_layers) fetch(l + p.slots);  // into the slot this layer has left
        cur ^= 1;
    }
    if (*(volatile int *)&abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies in flight land
        return;
    }

    // columns [0, n_actions) are logits, a further one is the state value
    const int A = p.n_actions;
    for (int i = tid; i < kRows * A; i += 32 * kMlpWarps) {
        const int r = i / A, c = i - r * A;
        if (row0 + r < B) logits[(long long)row0 * A + i] = s_logits[r][c];
    }
    if (value && tid < kRows && row0 + tid < B) value[row0 + tid] = s_logits[tid][A];
    // sampling: one thread per row (at most 32 actions)
    if (tid < kRows && row0 + tid < B) {
        const float *z = s_logits[tid];
        float m = z[0];
        int amax = 0;
        for (int i = 1; i < A; ++i)
            if (z[i] > m) {
                m = z[i];
                amax = i;
            }
        float s = 0.f;  // sum over all but the first maximal term, which is exp(0) = 1
        for (int i = 0; i < A; ++i)
            if (i != amax) s += expf(z[i] - m);
        const float l1p = log1pf(s), uu = u[row0 + tid];
        float cdf = 0.f, lp_a = 0.f, h = 0.f;
        int a = -1;
        for (int i = 0; i < A; ++i) {
            const float lp = (z[i] - m) - l1p, pi = expf(lp);
            if (pi > 0.f) h -= pi * lp;
            cdf += pi;
            if (a < 0 && uu < cdf) {
                a = i;
                lp_a = lp;
            }
        }
        if (a < 0) {
            a = A - 1;
            lp_a = (z[a] - m) - l1p;
        }
        actions[row0 + tid] = a;
        logp[row0 + tid] = lp_a;
        if (entropy) entropy[row0 + tid] = h;
    }
}

// Builds the fused plan when the policy qualifies; `used` says whether it did.
accerl_status build_mlp_plan(accerl_policy *p, const accerl_layer_desc *layers, int n_layers,
                             bool *used)
{
    *used = false;
    if (p->in_kind != ACCERL_IN_F32 || n_layers > kMaxLayers || p->n_out > 32) return ACCERL_OK;
    if (round_up(p->in_c, 4) > kMaxWidth) return ACCERL_OK;
    for (int i = 0; i < n_layers; ++i)
        if (layers[i].kind != ACCERL_FC || layers[i].out_c > kMaxWidth ||
            (layers[i].flags & ACCERL_RELU_IN) || !std::isfinite(1.0f / layers[i].s_out))  // (the kernel multiplies by it)
            return ACCERL_OK;
    auto prm = std::make_shared<MlpFusedParams>();
    memset(prm.get(), 0, sizeof(MlpFusedParams));
    prm->n_layers = n_layers;
    prm->in_dim = p->in_c;
    prm->n_actions = p->n_actions;
    prm->s_input = p->s_input;
    int k_in = p->in_c;
    for (int i = 0; i < n_layers; ++i) {
        const accerl_layer_desc &d = layers[i];
        const bool last = i == n_layers - 1;
        // hidden layers compute (zero) codes up to the next layer's K step
        const int KT = (k_in + 31) / 32, NT = last ? (d.out_c + 7) / 8 : round_up(d.out_c, 32) / 8;
        std::vector<int8_t> packed((size_t)NT * (KT * 256 + 64), 0);
        for (int o = 0; o < d.out_c; ++o)
            for (int k = 0; k < k_in; ++k) {
                // lane 4 g + q holds column g, bytes 4 q .. 4 q + 3 of both 16-byte halves of the K step
                const int in_step = k % 32, lane = 4 * (o % 8) + (in_step % 16) / 4;
                packed[(((size_t)(o / 8) * KT + k / 32) * 32 + lane) * 8 + 4 * (in_step / 16) + in_step % 4] =
                    d.w[(size_t)o * k_in + k];
            }
        float *ks = reinterpret_cast<float *>(packed.data() + (size_t)NT * KT * 256), *bs = ks + 8 * NT;
        for (int o = 0; o < d.out_c; ++o) {
            volatile float k = d.s_in * d.s_w[o];  // one fp32 rounding, never contracted
            ks[o] = k;
            bs[o] = d.bias[o];
        }
        void *dev = nullptr;
        accerl_status st = upload_bytes(p, packed.data(), packed.size(), &dev);
        if (st != ACCERL_OK) return st;
        volatile float inv = 1.0f / d.s_out;
        prm->block[i] = (const uint8_t *)dev;
        prm->block_bytes[i] = (uint32_t)packed.size();
        prm->kt[i] = KT;
        prm->nt[i] = NT;
        prm->n[i] = d.out_c;
        prm->inv_s_out[i] = inv;
        prm->relu[i] = (d.flags & ACCERL_RELU_OUT) != 0;
        prm->s_out[i] = d.s_out;
        if ((p->flags & ACCERL_FLAG_KEEP_ACTIVATIONS) && i + 1 < n_layers) {
            prm->tap[i] = p->bufs[p->layers[i].out_buf].ptr;
            prm->tap_pitch[i] = p->layers[i].out_cp;
        }
        k_in = d.out_c;
    }
    if (p->flags & ACCERL_FLAG_KEEP_ACTIVATIONS) {
        prm->tap_in = p->bufs[p->layers[0].in_buf].ptr;
        prm->tap_in_pitch = p->in_cp;
    }
    // Every layer has a place of its own in shared memory while two CTAs still fit an SM; deeper networks
    // pass through two slots, layer l + 2 fetched when layer l is done.
    uint32_t all = 0, widest = 0;
    for (int i = 0; i < n_layers; ++i) {
        all += prm->block_bytes[i];
        widest = std::max(widest, prm->block_bytes[i]);
    }
    prm->slots = all <= 84 * 1024 || n_layers <= 2 ? n_layers : 2;
    for (int i = 0, off = 0; i < n_layers; ++i) {
        prm->slot_off[i] = prm->slots == n_layers ? (uint32_t)off : (uint32_t)(i & 1) * widest;
        off += (int)prm->block_bytes[i];
    }
    prm->smem_bytes = prm->slots == n_layers ? all : 2 * widest;
    prm->status = p->status_word;
    p->mlp = prm;
    Step s;
    s.kind = Step::MLP_FUSED;
    s.kernel = "mlp_fused_kernel";
    s.covers = "ingest+layers 0-" + std::to_string(n_layers - 1) + "+sample";
    if (n_layers == 1) s.covers = "ingest+layer 0+sample";
    p->steps.assign(1, s);
    *used = true;
    return ACCERL_OK;
}

cudaError_t launch_mlp_fused(const accerl_policy *p, const float *obs, const float *u, int B,
                             float *logits, int32_t *actions, float *logp, float *value, float *entropy,
                             cudaStream_t st)
{
    const MlpFusedParams &prm = *p->mlp;
    auto go = [&](auto kernel, int rows) -> cudaError_t {
        cudaError_t e = allow_smem((const void *)kernel, prm.smem_bytes);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((B + rows - 1) / rows));
        cfg.blockDim = dim3(32 * kMlpWarps);
        cfg.dynamicSmemBytes = prm.smem_bytes;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, prm, obs, u, B, logits, actions, logp, value, entropy);
    };
    // 32 states per CTA once 16 would give every SM more than the two CTAs it holds at once: the weights are
    // then read half as often
    return B > 32 * p->sm_count ? go(mlp_fused_kernel<2>, 32) : go(mlp_fused_kernel<1>, 16);
}

}  // namespace accerl
