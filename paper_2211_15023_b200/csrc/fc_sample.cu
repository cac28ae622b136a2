// Last fully connected layer and the sampler in one launch: logits = fmaf((float)acc, k, b) for at
// most 32 actions, then log-softmax, inverse-CDF sampling and the behaviour log-prob of the drawn
// action.  The layer is tiny (K <= 1024, A <= 32), so a tensor-core launch plus a sampler launch
// spend most of their time starting and draining; here a warp owns two states at a time, lane j
// accumulates action j with dp4a from weights held in shared memory as [K/4][32] words, and the
// logits never leave registers before they are sampled (they are still written out: they are an
// output of the step).
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <vector>

#include "epilogue.cuh"
#include "internal.h"
#include "warp_sample.cuh"

namespace accerl {

namespace {

constexpr int kFsWarps = 8;

// EXTRAS: the states may be routed (Route); the layer may have one output column more than actions, the state value V(s) (lane A;
// no part of the softmax), and the entropy of the action distribution may be asked for.
template <bool EXTRAS>
__global__ void __launch_bounds__(32 * kFsWarps)
fc_sample_kernel(const FcSampleParams q, const float *__restrict__ u, int B_all, const Route route,
                 float *__restrict__ logits, int32_t *__restrict__ actions, float *__restrict__ logp,
                 float *__restrict__ value, float *__restrict__ entropy)
{
    extern __shared__ __align__(16) int32_t fs_smem[];
    const int K4 = q.k4, A = q.n_actions;
    int32_t *s_w = fs_smem;            // [K4][32]
    int32_t *s_x = fs_smem + K4 * 32;  // [warp][2][K4]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t *x0 = s_x + warp * 2 * K4, *x1 = x0 + K4;
    const bool live = lane < A;
    int B = B_all;
    const bool has_col = EXTRAS ? lane < q.n_out : live;  // a column of the layer (action or value)
    const long long stride = (long long)gridDim.x * kFsWarps;
    long long pair = (long long)blockIdx.x * kFsWarps + warp;
    // The first rows, the weights and the scales are all fetched before anything waits: the
    // kernel is a chain of a few dependent memory round trips, not a throughput problem.
    uint4 r0[2], r1[2];  // K <= 1024: at most two 16-byte pieces of a row per lane
    auto fetch = [&](long long pr) {
        const long long row0 = 2 * pr, row1 = row0 + 1;
        const uint4 *g0 = reinterpret_cast<const uint4 *>(q.x + row0 * q.pitch);
        const uint4 *g1 = reinterpret_cast<const uint4 *>(q.x + row1 * q.pitch);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = lane + 32 * j;
            const bool in = i < K4 / 4 && row0 < B;
            r0[j] = in ? __ldg(g0 + i) : make_uint4(0, 0, 0, 0);
            r1[j] = (in && row1 < B) ? __ldg(g1 + i) : make_uint4(0, 0, 0, 0);
        }
    };
    // Programmatic dependent launch: the weights and scales do not depend on the previous launch,
    // so they are fetched while it drains; the rows it wrote are read after the wait.  (No early
    // trigger of its own: a next step's first layer that starts while this kernel still runs takes
    // its SMs' issue slots just to wait -- measured 194 against 177 us per Nature-CNN step.)
    const float ks = has_col ? q.kscale[lane] : 0.f, bs = has_col ? q.bias[lane] : 0.f;
    {
        const uint4 *gw = reinterpret_cast<const uint4 *>(q.w);
        uint4 *sw = reinterpret_cast<uint4 *>(s_w);
        for (int i = threadIdx.x; i < K4 * 8; i += blockDim.x) sw[i] = __ldg(gw + i);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (EXTRAS) B = routed_batch(route, B_all);
    fetch(pair);
    __syncthreads();
    for (; 2 * pair < B; pair += stride) {
        const long long row0 = 2 * pair, row1 = row0 + 1;
        const bool has1 = row1 < B;
        // where the results go, and the states' uniforms
        const long long out0 = EXTRAS ? routed_row(route, (int)row0) : row0, out1 = EXTRAS && has1 ? routed_row(route, (int)row1) : row1;
        const float u0 = u[out0], u1 = has1 ? u[out1] : 2.f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = lane + 32 * j;
            if (i < K4 / 4) {
                reinterpret_cast<uint4 *>(x0)[i] = r0[j];
                reinterpret_cast<uint4 *>(x1)[i] = r1[j];
            }
        }
        __syncwarp();
        fetch(pair + stride);  // the next round's rows travel while this one computes
        int acc0 = 0, acc1 = 0;
#pragma unroll 4
        for (int k = 0; k < K4; k += 4) {
            const uint4 a0 = *reinterpret_cast<const uint4 *>(x0 + k);
            const uint4 a1 = *reinterpret_cast<const uint4 *>(x1 + k);
            const int w0 = s_w[k * 32 + lane], w1 = s_w[(k + 1) * 32 + lane];
            const int w2 = s_w[(k + 2) * 32 + lane], w3 = s_w[(k + 3) * 32 + lane];
            acc0 = __dp4a((int)a0.x, w0, acc0);
            acc1 = __dp4a((int)a1.x, w0, acc1);
            acc0 = __dp4a((int)a0.y, w1, acc0);
            acc1 = __dp4a((int)a1.y, w1, acc1);
            acc0 = __dp4a((int)a0.z, w2, acc0);
            acc1 = __dp4a((int)a1.z, w2, acc1);
            acc0 = __dp4a((int)a0.w, w3, acc0);
            acc1 = __dp4a((int)a1.w, w3, acc1);
        }
        __syncwarp();  // the staged rows are overwritten in the next round
        const float z0 = epilogue_float(acc0, ks, bs, false), z1 = epilogue_float(acc1, ks, bs, false);
        if (live) {
            logits[out0 * A + lane] = z0;
            if (has1) logits[out1 * A + lane] = z1;
        }
        if (EXTRAS && value && lane == A && A < q.n_out) {
            value[out0] = z0;
            if (has1) value[out1] = z1;
        }
        int a;
        float lpa, h = 0.f;
        if (EXTRAS && entropy) warp_sample<true>(z0, live, u0, A, lane, a, lpa, h);
        else warp_sample<false>(z0, live, u0, A, lane, a, lpa, h);
        if (lane == 0) {
            actions[out0] = a;
            logp[out0] = lpa;
            if (EXTRAS && entropy) entropy[out0] = h;
        }
        if (EXTRAS && entropy) warp_sample<true>(z1, live, u1, A, lane, a, lpa, h);
        else warp_sample<false>(z1, live, u1, A, lane, a, lpa, h);
        if (lane == 0 && has1) {
            actions[out1] = a;
            logp[out1] = lpa;
            if (EXTRAS && entropy) entropy[out1] = h;
        }
    }
}

// ---------------------------------------------------------------------------------------
// hidden fully connected layer, last layer and sampler in one launch, for small batches
// ---------------------------------------------------------------------------------------
// A hidden layer of 256 or 512 outputs on up to a few hundred states is a stream of weights (1.6 MB for
// the Nature-CNN) against hardly any rows: as 128-row tiles of the big tensor pipe it occupies 32 SMs and
// took about 10 us, and the last layer with the sampler another launch after it.  Here a cluster of eight
// CTAs owns 16 or 32 states; CTA c computes columns c * N / 8 .. of the hidden layer on warp-level int8
// tensor instructions, sixteen warps with a share of K each (operands straight from L2 to registers, in
// 64-byte pieces of K so that every load instruction moves whole sectors), adds the partial sums through
// shared memory, requantises, and hands every state's codes to the CTA that finishes it: two or four
// states each, last layer by dp4a, softmax, draw.  The weights of the last layer are in registers before
// the previous launch is done.
constexpr int kHeadWarps = 16, kHeadCluster = 8;

__device__ __forceinline__ void head_mma(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// MT: 16-state tiles of a cluster; NT: 8-column tiles of a CTA (N = 64 * NT hidden outputs)
template <int MT, int NT>
__global__ void __launch_bounds__(32 * kHeadWarps, 1)
fc_hidden_fc_sample_kernel(const __grid_constant__ FcHeadParams h, const __grid_constant__ FcSampleParams q, const float *__restrict__ u, int B_all,
                           const Route route,
                           float *__restrict__ logits, int32_t *__restrict__ actions, float *__restrict__ logp,
                           float *__restrict__ value, float *__restrict__ entropy)
{
    constexpr int kRows = 16 * MT, kCols = 8 * NT, kN = kCols * kHeadCluster;
    constexpr int kOwn = kRows / kHeadCluster;          // states a CTA finishes
    constexpr int kSlices = kHeadWarps / kOwn;          // warps that share one of them
    constexpr int kWords = kN / 4 / kSlices;            // words of its codes each takes
    extern __shared__ __align__(16) int32_t head_smem[];  // partial sums [warp][kRows][kCols]
    __shared__ __align__(16) uint32_t codes[kOwn][kN / 4];
    __shared__ int s_z[kOwn][kSlices][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int rank = (int)cooperative_groups::this_cluster().block_rank();
    const int row0 = (int)(blockIdx.x / kHeadCluster) * kRows;

    // what does not depend on the previous launch
    const int own = warp / kSlices, slice = warp % kSlices;
    int w2[kWords];
#pragma unroll
    for (int k = 0; k < kWords; ++k) w2[k] = __ldg(q.w + (slice * kWords + k) * 32 + lane);
    const bool has_col = lane < q.n_out;
    const float ks2 = has_col ? q.kscale[lane] : 0.f, bs2 = has_col ? q.bias[lane] : 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int B = routed_batch(route, B_all);
    if (row0 >= B) return;  // the whole cluster

    // ---- hidden layer: this warp's pieces of K
    int acc[MT][NT][4] = {};
    const int8_t *xr[2 * MT];
#pragma unroll
    for (int m = 0; m < 2 * MT; ++m) xr[m] = h.x + (long long)min(row0 + 8 * m + g, B - 1) * h.K + 16 * t;
    const uint4 *wp = h.w + (size_t)rank * NT * 32 + lane;  // [piece][N / 8][lane]
#pragma unroll 2
    for (int p = warp; p < h.pieces; p += kHeadWarps) {
        uint4 a[2 * MT], b[NT];
        const bool in = 64 * p + 16 * t < h.K;  // (K is a multiple of 16; the weights are padded with zeros)
#pragma unroll
        for (int m = 0; m < 2 * MT; ++m) a[m] = in ? __ldcg(reinterpret_cast<const uint4 *>(xr[m] + 64 * p)) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int n = 0; n < NT; ++n) b[n] = __ldg(wp + ((size_t)p * (NT * kHeadCluster) + n) * 32);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                head_mma(acc[m][n], a[2 * m].x, a[2 * m + 1].x, a[2 * m].y, a[2 * m + 1].y, b[n].x, b[n].y);
                head_mma(acc[m][n], a[2 * m].z, a[2 * m + 1].z, a[2 * m].w, a[2 * m + 1].w, b[n].z, b[n].w);
            }
    }
    // (no early trigger: the next launch waits for this one as a whole)
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                *reinterpret_cast<int2 *>(head_smem + (warp * kRows + 16 * m + 8 * r + g) * kCols + 8 * n + 2 * t) =
                    make_int2(acc[m][n][2 * r], acc[m][n][2 * r + 1]);
    cooperative_groups::this_cluster().sync();  // also: every CTA of the cluster has started, its shared memory may be written
    for (int i = threadIdx.x; i < kRows * kCols / 2; i += 32 * kHeadWarps) {
        const int r = i / (kCols / 2), c = 2 * (i - r * (kCols / 2));
        int2 s = make_int2(0, 0);
#pragma unroll
        for (int w = 0; w < kHeadWarps; ++w) {
            const int2 v = *reinterpret_cast<const int2 *>(head_smem + (w * kRows + r) * kCols + c);
            s.x += v.x;
            s.y += v.y;
        }
        const int col = rank * kCols + c;
        const float2 k = __ldg(reinterpret_cast<const float2 *>(h.kscale + col)), b = __ldg(reinterpret_cast<const float2 *>(h.bias + col));
        uint32_t code = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j)
            code |= (uint32_t)(uint8_t)requant(epilogue_float(j ? s.y : s.x, j ? k.y : k.x, j ? b.y : b.x, h.relu != 0), h.s_out) << (8 * j);
        uint16_t *mine = reinterpret_cast<uint16_t *>(&codes[r % kOwn][0]) + col / 2;
        *cooperative_groups::this_cluster().map_shared_rank(mine, (unsigned)(r / kOwn)) = (uint16_t)code;
        if (h.tap && row0 + r < B) *reinterpret_cast<uint16_t *>(h.tap + (long long)(row0 + r) * kN + col) = (uint16_t)code;
    }
    cooperative_groups::this_cluster().sync();
    // ---- last layer: lane = column, a slice of K per warp
    {
        int z = 0;
        const uint4 *x = reinterpret_cast<const uint4 *>(&codes[own][slice * kWords]);
#pragma unroll
        for (int k = 0; k < kWords / 4; ++k) {
            const uint4 v = x[k];
            z = __dp4a((int)v.x, w2[4 * k], z);
            z = __dp4a((int)v.y, w2[4 * k + 1], z);
            z = __dp4a((int)v.z, w2[4 * k + 2], z);
            z = __dp4a((int)v.w, w2[4 * k + 3], z);
        }
        s_z[own][slice][lane] = z;
    }
    __syncthreads();
    const int row = row0 + rank * kOwn + own;
    if (slice != 0 || row >= B) return;
    int zi = 0;
#pragma unroll
    for (int s = 0; s < kSlices; ++s) zi += s_z[own][s][lane];
    const float z = epilogue_float(zi, ks2, bs2, false);
    const int A = q.n_actions, out = routed_row(route, row);
    const bool live = lane < A;
    if (live) logits[(long long)out * A + lane] = z;
    if (value && lane == A && A < q.n_out) value[out] = z;
    int a;
    float lpa, hh = 0.f;
    if (entropy) warp_sample<true>(z, live, u[out], A, lane, a, lpa, hh);
    else warp_sample<false>(z, live, u[out], A, lane, a, lpa, hh);
    if (lane == 0) {
        actions[out] = a;
        logp[out] = lpa;
        if (entropy) entropy[out] = hh;
    }
}

}  // namespace

// Can layer i (the last one) run fused with the sampler?  Its input must be a plain [B][K] int8
// matrix written by a fully connected layer.
bool fc_sample_fits(const accerl_policy *p, const accerl_layer_desc *layers, int n_layers, int i)
{
    if (i != n_layers - 1 || i < 1) return false;
    const accerl_layer_desc &d = layers[i];
    const LayerPlan &L = p->layers[i];
    if (d.kind != ACCERL_FC || !(d.flags & ACCERL_LOGITS) || layers[i - 1].kind != ACCERL_FC) return false;
    if ((d.flags & ACCERL_RELU_IN) && !(layers[i - 1].flags & ACCERL_RELU_OUT)) return false;
    const int K = L.in_c;
    return L.in_h == 1 && L.in_w == 1 && L.in_cp == L.in_c && K % 16 == 0 && K >= 16 && K <= 1024 &&
           d.out_c <= 32;
}

// Packs the weights and fills the step; x is the layer's input matrix with rows of `pitch` bytes.
accerl_status build_fc_sample(accerl_policy *p, const accerl_layer_desc &d, int layer, const int8_t *x,
                              int pitch, Step *out)
{
    const LayerPlan &L = p->layers[layer];
    const int K = L.in_c, K4 = K / 4;
    std::vector<int32_t> words((size_t)K4 * 32, 0);
    for (int o = 0; o < d.out_c; ++o)
        for (int k = 0; k < K; ++k)
            words[(size_t)(k / 4) * 32 + o] |=
                (int32_t)((uint32_t)(uint8_t)d.w[(size_t)o * K + k] << (8 * (k % 4)));
    void *dev = nullptr;
    accerl_status st = upload_bytes(p, words.data(), words.size() * 4, &dev);
    if (st != ACCERL_OK) return st;
    FcSampleParams &q = p->fc_sample;
    q.x = x;
    q.pitch = pitch;
    q.k4 = K4;
    q.n_actions = p->n_actions;
    q.n_out = d.out_c;
    q.w = (const int32_t *)dev;
    q.kscale = L.kscale;
    q.bias = L.bias;
    out->kind = Step::FC_SAMPLE;
    out->layer = layer;
    out->kernel = "fc_sample_kernel";
    out->covers = "layer " + std::to_string(layer) + "+sample";
    return ACCERL_OK;
}

// Clusters of eight that find their SMs at once: 15 on 148 SMs; one less, should another chip's SMs lie less well
static int head_clusters(int sm_count) { return sm_count / 10; }

// Do the hidden layer `i` and the last one behind it run as that launch?  Handles for more states end in
// tiles of 128 (fc_tile.cu), which read the weights less often, or in two launches.  The line lies where this
// launch's clusters no longer fit the chip at once, with 16 states each for 512 outputs, 32 for 256: 224 and 448
// states on 148 SMs (us per step, this launch / tiles: 512 outputs of 3136 inputs 15.4 / 19.3 at 160 states, 22.1 /
// 20.3 at 256; 256 of 1568 11.0 / 13.6, 15.9 / 17.4 at 448, 22.3 / 18.7 at 640).  A handle made for one state, as
// accerl_policy_act_noalloc asks for, has this launch at every batch of its fixed workspace.
bool fc_head_fits(const accerl_policy *p, const accerl_layer_desc *layers, int n_layers, int i)
{
    if (i != n_layers - 2 || i < 1 || unfuse_for_taps(p) || !fc_sample_fits(p, layers, n_layers, i + 1)) return false;
    const accerl_layer_desc &d = layers[i];
    const LayerPlan &L = p->layers[i];
    return d.kind == ACCERL_FC && (d.out_c == 256 || d.out_c == 512) && p->max_batch <= head_clusters(p->sm_count) * (d.out_c == 512 ? 16 : 32) &&
           L.in_cp == L.in_c && (L.in_h * L.in_w * L.in_cp) % 16 == 0;
}

// x: the hidden layer's input rows; its weights in (y, x, c) order are L.host_rows
accerl_status build_fc_head(accerl_policy *p, const accerl_layer_desc *layers, int i, const int8_t *x, Step *out)
{
    const accerl_layer_desc &d = layers[i];
    const LayerPlan &L = p->layers[i];
    const int K = L.in_h * L.in_w * L.in_cp, N = d.out_c, pieces = (K + 63) / 64;
    // [piece][column / 8][lane 4 g + t]: bytes 16 t .. 16 t + 15 of the piece, column g
    const int8_t *rows = L.host_rows;
    void *dev = nullptr, *host = nullptr;
    accerl_status st = upload_room(p, (size_t)pieces * N * 64, &host, &dev);
    if (st != ACCERL_OK) return st;
    int8_t *at = (int8_t *)host;
    for (int k0 = 0; k0 < K; k0 += 64)
        for (int o = 0; o < N; ++o, at += 64)
            for (int k = k0; k < K && k < k0 + 64; k += 16) memcpy(at + (k - k0), rows + (size_t)o * K + k, 16);
    FcHeadParams &h = p->fc_head;
    h.x = x;
    h.w = (const uint4 *)dev;
    h.K = K;
    h.pieces = pieces;
    h.N = N;
    h.kscale = L.kscale;
    h.bias = L.bias;
    h.s_out = L.s_out;
    h.relu = (d.flags & ACCERL_RELU_OUT) != 0;
    h.tap = (p->flags & ACCERL_FLAG_KEEP_ACTIVATIONS) ? p->bufs[L.out_buf].ptr : nullptr;
    Step last;
    if ((st = build_fc_sample(p, layers[i + 1], i + 1, nullptr, N, &last)) != ACCERL_OK) return st;
    out->kind = Step::FC_HEAD;
    out->kernel = "fc_hidden_fc_sample_kernel";
    out->covers = "layers " + std::to_string(i) + "-" + std::to_string(i + 1) + "+sample";
    return ACCERL_OK;
}

cudaError_t launch_fc_head(const FcHeadParams &h, const FcSampleParams &q, const float *u, int B, float *logits,
                           int32_t *actions, float *logp, float *value, float *entropy, const Route &route, int sm_count,
                           cudaStream_t st)
{
    auto go = [&](auto kernel, int rows) -> cudaError_t {
        const size_t smem = sizeof(int) * (size_t)kHeadWarps * rows * (h.N / kHeadCluster);
        cudaError_t e = allow_smem((const void *)kernel, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((B + rows - 1) / rows * kHeadCluster));
        cfg.blockDim = dim3(32 * kHeadWarps);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = kHeadCluster;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        return cudaLaunchKernelEx(&cfg, kernel, h, q, u, B, route, logits, actions, logp, value, entropy);
    };
    // 16 states per cluster while their clusters fit the chip at once: with 16 clusters, at 256 states, a step of the
    // narrow network took 15.4 us, with half as many 12.9
    const bool two = ((route.count ? route.expect : B) + 15) / 16 > head_clusters(sm_count);
    if (h.N == 512) return two ? go(fc_hidden_fc_sample_kernel<2, 8>, 32) : go(fc_hidden_fc_sample_kernel<1, 8>, 16);
    return two ? go(fc_hidden_fc_sample_kernel<2, 4>, 32) : go(fc_hidden_fc_sample_kernel<1, 4>, 16);
}

cudaError_t launch_fc_sample(const FcSampleParams &q, const float *u, int B, float *logits,
                             int32_t *actions, float *logp, float *value, float *entropy, const Route &route,
                             int sm_count, cudaStream_t st)
{
    const int per_block = 2 * kFsWarps;
    long long blocks = ((long long)B + per_block - 1) / per_block;
    if (blocks > 4LL * sm_count) blocks = 4LL * sm_count;
    const size_t smem = (size_t)q.k4 * 4 * (32 + 2 * kFsWarps);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(32 * kFsWarps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool extras = value || entropy || q.n_out != q.n_actions || route.count;
    cudaError_t e = extras ? cudaLaunchKernelEx(&cfg, fc_sample_kernel<true>, q, u, B, route, logits, actions, logp, value, entropy)
                           : cudaLaunchKernelEx(&cfg, fc_sample_kernel<false>, q, u, B, route, logits, actions, logp,
                                                (float *)nullptr, (float *)nullptr);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace accerl
