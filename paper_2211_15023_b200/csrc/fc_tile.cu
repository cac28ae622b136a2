// Hidden fully connected layer, last layer and sampler in one launch, for batches of a few hundred states
// to one wave of the chip: the tensor-core sibling of fc_hidden_fc_sample_kernel.
//
// The hidden layer is a 128-state tile per cluster, its 256 or 512 outputs split over the cluster's CTAs:
// each streams its columns of the weights and the tile's rows of K through shared memory into one
// accumulator, requantises, and hands every state's codes to the CTA that finishes it (128 / C states
// each): last layer on warp-level int8 tensor instructions, K split over the warps, then softmax and draw,
// a warp per state.  The hidden activations never leave the chip.
//
// What bounds it: the operands' way from L2 (a state tile's rows are read by every CTA of its cluster, the
// weights by every cluster), and below some 2000 states the chain load - contract - exchange - sample.  As
// two launches (a contraction whose output goes through L2 to fc_sample_kernel) the tail cost a second
// launch, a drain and a fill.  A whole step, two launches / this one: 512 outputs of 3136 inputs 40.9 / 36.6 us
// for 1237 states, 56.9 / 51.1 for 2048, 139.9 / 136.8 for 8192; 256 of 1568 23.5 / 18.9 for 700, 28.8 / 25.6 for
// 1237, 111.7 / 107.9 for 8192.
//
// Every wait is bounded; a role whose wait gives up sets the status word and goes on.
#include <cooperative_groups.h>
#include <cuda.h>
#include <string.h>

#include <vector>

#include "internal.h"
#include "tc_image.cuh"
#include "warp_sample.cuh"

namespace accerl {

namespace {

constexpr int kTileThreads = 512;
constexpr int kPartPitch = 40;  // ints between rows of partial sums: eight rows' column pairs fill the banks

// NT: hidden columns of a CTA, C: CTAs of a cluster
template <int NT, int C>
struct TileSizes {
    static constexpr int n = NT * C, rows = 128 / C, stage = 128 * 128 + NT * 128, stages = 192 * 1024 / stage < 8 ? 192 * 1024 / stage : 8;
    static constexpr int code_pitch = n + 16;  // (16-byte pieces of eight rows fill the banks)
    static constexpr int parts = (rows * code_pitch + 1023) & ~1023;
    static constexpr int mtiles = rows / 16, ksplit = 16 / mtiles, ksteps = n / 32, per_warp = (ksteps + ksplit - 1) / ksplit;
    static constexpr size_t smem = 1024 + (size_t)stages * stage;
    // the codes and the partial sums lie where the operands were
    static_assert(parts + ksplit * rows * kPartPitch * 4 <= stages * stage && rows % 16 == 0 && NT % 32 == 0, "layout");
};

struct __align__(8) TileBars {
    uint64_t full[8], empty[8], acc;
    uint32_t tmem_base;
    int abort_flag;
};

__device__ __forceinline__ void tile_mma(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int NT, int C>
__global__ void __launch_bounds__(kTileThreads, 1)
fc_tile_fc_sample_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ FcTileParams h,
                         const __grid_constant__ FcSampleParams q, const float *__restrict__ u, int B_all, const Route route,
                         float *__restrict__ logits, int32_t *__restrict__ actions, float *__restrict__ logp,
                         float *__restrict__ value, float *__restrict__ entropy)
{
    using S = TileSizes<NT, C>;
    constexpr uint32_t kCols = NT;  // of tensor memory
    extern __shared__ __align__(1024) uint8_t tile_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)tile_smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ TileBars bars;
    __shared__ __align__(16) float s_k[NT], s_b[NT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int rank = C == 1 ? 0 : (int)(blockIdx.x % C), row0 = (int)(blockIdx.x / C) * 128;
    volatile int *abort_flag = &bars.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::stages; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 1);
            mbar_init(smem_u32(&bars.empty[s]), 1);
        }
        mbar_init(smem_u32(&bars.acc), 1);
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)), "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if ((int)threadIdx.x < NT) {
        s_k[threadIdx.x] = __ldg(h.k + rank * NT + threadIdx.x);
        s_b[threadIdx.x] = __ldg(h.b + rank * NT + threadIdx.x);
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = bars.tmem_base, base = smem_u32(smem), full0 = smem_u32(&bars.full[0]), empty0 = smem_u32(&bars.empty[0]);
    const int chunks = h.chunks;
    auto load_w = [&](int ch) {
        const uint32_t s = (uint32_t)(ch % S::stages);
        mbar_expect_tx(full0 + 8 * s, (uint32_t)S::stage);
        bulk_load(base + s * S::stage + 128 * 128, h.w + ((size_t)ch * S::n + rank * NT) * 128, NT * 128, full0 + 8 * s);
    };
    // What does not depend on the previous launch: the first stages' weights (unless there may turn out to be no
    // state for this cluster) and the last layer's, this warp's K steps and all columns
    const bool early = !route.count;
    if (warp == 0 && early && elect_one())
        for (int ch = 0; ch < S::stages && ch < chunks; ++ch) load_w(ch);
    __syncwarp();
    const int mt = warp % S::mtiles, sp = warp / S::mtiles;
    uint32_t wb[S::per_warp][4][2];
#pragma unroll
    for (int j = 0; j < S::per_warp; ++j) {
        const int ks = sp + j * S::ksplit;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) wb[j][n][i] = ks < S::ksteps ? (uint32_t)__ldg(q.w + (ks * 8 + 4 * i + t) * 32 + 8 * n + g) : 0u;
    }
    const bool has_col = lane < q.n_out;
    const float ks2 = has_col ? q.kscale[lane] : 0.f, bs2 = has_col ? q.bias[lane] : 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int B = routed_batch(route, B_all);

    if (row0 < B) {  // (the same for the whole cluster)
        // ---- hidden layer
        if (warp == 0) {
            for (int ch = 0; ch < chunks; ++ch) {
                const uint32_t s = (uint32_t)(ch % S::stages);
                if (ch >= S::stages) image_wait(empty0 + 8 * s, (uint32_t)((ch / S::stages - 1) & 1), abort_flag, h.status, 1);
                if (elect_one()) {
                    if (!early || ch >= S::stages) load_w(ch);
                    tma_load_2d(base + s * S::stage, &map_x, ch * 128, row0, full0 + 8 * s);
                }
                __syncwarp();
            }
        } else if (warp == 1) {
            for (int ch = 0; ch < chunks; ++ch) {
                const uint32_t s = (uint32_t)(ch % S::stages);
                image_wait(full0 + 8 * s, (uint32_t)((ch / S::stages) & 1), abort_flag, h.status, 8);
                fence_after();
                if (elect_one()) {
                    const uint64_t a = make_desc(base + s * S::stage, 128), b = make_desc(base + s * S::stage + 128 * 128, 128);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) mma_i8(tmem, a + 2 * ks, b + 2 * ks, idesc_for(NT), (uint32_t)(ch | ks));
                    mma_commit(empty0 + 8 * s);
                    if (ch == chunks - 1) mma_commit(smem_u32(&bars.acc));
                }
                __syncwarp();
            }
        }
        image_wait(smem_u32(&bars.acc), 0, abort_flag, h.status, 16);
        fence_after();
        // ---- codes, to the CTA that finishes the state
        constexpr int kPieces = NT / 16, kMine = (kPieces + 3) / 4;
        const int wg = warp >> 2, r = (warp & 3) * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        uint4 code[kMine];
#pragma unroll
        for (int j = 0; j < kMine; ++j) {
            const int p = wg * kMine + j;
            if (p < kPieces) {
                int acc[16];
                tmem_ld16(tlane + 16 * p, acc);
                tmem_wait_ld();
                float ks[16], bs[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 kv = *reinterpret_cast<const float4 *>(&s_k[16 * p + 4 * i]), bv = *reinterpret_cast<const float4 *>(&s_b[16 * p + 4 * i]);
                    ks[4 * i] = kv.x; ks[4 * i + 1] = kv.y; ks[4 * i + 2] = kv.z; ks[4 * i + 3] = kv.w;
                    bs[4 * i] = bv.x; bs[4 * i + 1] = bv.y; bs[4 * i + 2] = bv.z; bs[4 * i + 3] = bv.w;
                }
                uint32_t w[4];
                if (h.affine) requant16_affine<false>(acc, ks, bs, w);
                else requant16_fastdiv<false>(acc, ks, bs, h.s_out, h.inv_s_out, w);
                code[j] = make_uint4(w[0], w[1], w[2], w[3]);
                if (h.relu) code[j] = relu16(code[j]);
                if (h.tap && row0 + r < B) *reinterpret_cast<uint4 *>(h.tap + (size_t)(row0 + r) * S::n + rank * NT + 16 * p) = code[j];
            }
        }
        auto cluster = cooperative_groups::this_cluster();
        if (C > 1) cluster.sync();  // every CTA's operands have been read: its codes may lie there
        else __syncthreads();
#pragma unroll
        for (int j = 0; j < kMine; ++j) {
            const int p = wg * kMine + j;
            if (p < kPieces) {
                uint4 *at = reinterpret_cast<uint4 *>(smem + (r % S::rows) * S::code_pitch + rank * NT + 16 * p);
                if (C > 1) at = cluster.map_shared_rank(at, (unsigned)(r / S::rows));
                *at = code[j];
            }
        }
        if (C > 1) cluster.sync();
        else __syncthreads();
        // ---- last layer: sixteen states and a share of K per warp
        int z[4][4] = {};
#pragma unroll
        for (int j = 0; j < S::per_warp; ++j) {
            const int ks = sp + j * S::ksplit;
            if (ks < S::ksteps) {
                const uint32_t *x0 = reinterpret_cast<const uint32_t *>(smem + (16 * mt + g) * S::code_pitch) + ks * 8 + t;
                const uint32_t *x1 = x0 + 8 * S::code_pitch / 4;
                const uint32_t a0 = x0[0], a1 = x1[0], a2 = x0[4], a3 = x1[4];
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    if (8 * n < q.n_out) tile_mma(z[n], a0, a1, a2, a3, wb[j][n][0], wb[j][n][1]);
            }
        }
        int *part = reinterpret_cast<int *>(smem + S::parts);
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                *reinterpret_cast<int2 *>(part + (sp * S::rows + 16 * mt + 8 * i + g) * kPartPitch + 8 * n + 2 * t) = make_int2(z[n][2 * i], z[n][2 * i + 1]);
        __syncthreads();
        // ---- a warp per state
        const int A = q.n_actions;
        const bool live = lane < A;
        for (int i = warp; i < S::rows; i += kTileThreads / 32) {
            const int row = row0 + rank * S::rows + i;
            if (row >= B) break;
            int zi = 0;
#pragma unroll
            for (int s = 0; s < S::ksplit; ++s) zi += part[(s * S::rows + i) * kPartPitch + lane];
            const float zf = epilogue_float(zi, ks2, bs2, false);
            const int out = routed_row(route, row);
            if (live) logits[(long long)out * A + lane] = zf;
            if (value && lane == A && A < q.n_out) value[out] = zf;
            int a;
            float lpa, hh = 0.f;
            if (entropy) warp_sample<true>(zf, live, u[out], A, lane, a, lpa, hh);
            else warp_sample<false>(zf, live, u[out], A, lane, a, lpa, hh);
            if (lane == 0) {
                actions[out] = a;
                logp[out] = lpa;
                if (entropy) entropy[out] = hh;
            }
        }
    }
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies in flight land
    fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

}  // namespace

// Do the hidden layer `i` and the last one behind it run as that launch?  Handles whose states, 128 by 128
// with 256 columns a CTA, are more than one wave stay with the two launches.
bool fc_tile_fits(const accerl_policy *p, const accerl_layer_desc *layers, int n_layers, int i)
{
    if (i != n_layers - 2 || i < 1 || unfuse_for_taps(p) || !p->requant[i].fast_div || !fc_sample_fits(p, layers, n_layers, i + 1)) return false;
    const accerl_layer_desc &d = layers[i];
    const LayerPlan &L = p->layers[i];
    return d.kind == ACCERL_FC && (d.out_c == 256 || d.out_c == 512) && L.in_cp == L.in_c && (L.in_h * L.in_w * L.in_cp) % 16 == 0 &&
           (long long)(p->max_batch + 127) / 128 * (d.out_c / 256) <= p->sm_count;
}

// x: the hidden layer's input rows; its weights in (y, x, c) order are L.host_rows
accerl_status build_fc_tile(accerl_policy *p, const accerl_layer_desc *layers, int i, const int8_t *x, Step *out)
{
    const accerl_layer_desc &d = layers[i];
    const LayerPlan &L = p->layers[i];
    const LayerRequant &rq = p->requant[i];
    const int K = L.in_h * L.in_w * L.in_cp, N = d.out_c, chunks = (K + 127) / 128;
    // [chunk of K][column][128 bytes under the 128-byte swizzle]
    const int8_t *rows = L.host_rows;
    void *w_host = nullptr, *w_dev = nullptr, *k_dev = nullptr, *b_dev = nullptr;
    accerl_status st = upload_room(p, (size_t)chunks * N * 128, &w_host, &w_dev);
    if (st != ACCERL_OK) return st;
    int8_t *at = (int8_t *)w_host;
    for (int k0 = 0; k0 < K; k0 += 128)
        for (int o = 0; o < N; ++o, at += 128)
            for (int k = k0; k < K && k < k0 + 128; k += 16) memcpy(at + ((((k - k0) / 16) ^ (o & 7)) << 4), rows + (size_t)o * K + k, 16);
    st = upload_bytes(p, rq.k.data(), (size_t)N * 4, &k_dev);
    if (st == ACCERL_OK) st = upload_bytes(p, rq.b.data(), (size_t)N * 4, &b_dev);
    if (st != ACCERL_OK) return st;
    p->fc_tile_a = ActivationMap{x, 1, K, K, 128, 128};
    if ((st = tc_make_map(p->fc_tile_map, x, p->max_batch, K, K, 128, 128)) != ACCERL_OK) return st;
    FcTileParams &h = p->fc_tile;
    h.w = (const uint8_t *)w_dev;
    h.chunks = chunks;
    h.N = N;
    h.k = (const float *)k_dev;
    h.b = (const float *)b_dev;
    h.s_out = L.s_out;
    h.inv_s_out = rq.inv_s_out;
    h.affine = rq.affine;
    h.relu = (d.flags & ACCERL_RELU_OUT) != 0;
    h.tap = (p->flags & ACCERL_FLAG_KEEP_ACTIVATIONS) ? p->bufs[L.out_buf].ptr : nullptr;
    h.status = p->status_word;
    Step last;
    if ((st = build_fc_sample(p, layers[i + 1], i + 1, nullptr, N, &last)) != ACCERL_OK) return st;
    out->kind = Step::FC_TILE;
    out->kernel = std::string("fc_tile_fc_sample_kernel") + (rq.affine ? "[single-fma requantiser verified]" : "[3-step divide verified]");
    out->covers = "layers " + std::to_string(i) + "-" + std::to_string(i + 1) + "+sample";
    return ACCERL_OK;
}

cudaError_t launch_fc_tile(const void *map_x, const FcTileParams &h, const FcSampleParams &q, const float *u, int B, float *logits,
                           int32_t *actions, float *logp, float *value, float *entropy, const Route &route, int sm_count,
                           cudaStream_t st)
{
    auto go = [&](auto cols, auto ctas) -> cudaError_t {
        constexpr int NT = decltype(cols)::value, C = decltype(ctas)::value;
        auto kernel = fc_tile_fc_sample_kernel<NT, C>;
        cudaError_t e = allow_smem((const void *)kernel, TileSizes<NT, C>::smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((B + 127) / 128 * C));
        cfg.blockDim = dim3(kTileThreads);
        cfg.dynamicSmemBytes = TileSizes<NT, C>::smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = C;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        CUtensorMap map;
        memcpy(&map, map_x, sizeof(map));
        return cudaLaunchKernelEx(&cfg, kernel, map, h, q, u, B, route, logits, actions, logp, value, entropy);
    };
    // As many CTAs per tile of states as the chip holds at once: 148 SMs take 15 clusters of eight (16 in two waves cost
    // 4 us of 60 at 2048 states), 33 of four, 74 of two.  One less of the larger ones, should another chip's SMs lie
    // less well; pairs lie wherever two SMs do.
    const int tiles = ((route.count ? route.expect : B) + 127) / 128;
    const int c = tiles <= sm_count / 10 ? 8 : tiles <= sm_count * 2 / 9 ? 4 : tiles <= sm_count / 2 || h.N == 512 ? 2 : 1;
    if (h.N == 512) return c == 8 ? go(OpIndex<64>(), OpIndex<8>()) : c == 4 ? go(OpIndex<128>(), OpIndex<4>()) : go(OpIndex<256>(), OpIndex<2>());
    return c == 8 ? go(OpIndex<32>(), OpIndex<8>()) : c == 4 ? go(OpIndex<64>(), OpIndex<4>()) : c == 2 ? go(OpIndex<128>(), OpIndex<2>())
                                                                                                       : go(OpIndex<256>(), OpIndex<1>());
}

}  // namespace accerl
