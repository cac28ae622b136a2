// The conv stack of the Atari networks (84 x 84 x 4 frames; 8 x 8 / 4, 4 x 4 / 2, 3 x 3; 32 / 64 / 64 or
// 16 / 32 / 32 channels) as one launch with its images resident in shared memory: uint8 frames in, the
// fully connected layer's int8 input rows out.
//
// One launch per layer (tc_conv1.cu, tc_conv.cu, tc_gemm.cu) keeps every unit busy with thousands of
// images, but a launch costs the host 2.5 us and the device a fill and a drain, and the paper's Actor has
// 160 states.  Here a CTA takes an image through all three layers: quantised 4 x 4 blocks of the frame,
// the first layer's output in space-to-depth form and the second layer's are operand rows of the next
// contraction in shared memory, all weights lie beside them.  Contractions are row-shifted implicit
// GEMMs as everywhere in this library: one GEMM row per grid position, taps at fixed row offsets; 441
// positions are four tiles of the first layer, 100 and 81 positions one tile of the other two.
//
// While there is an SM for every image a CTA is one context of sixteen warps (four warpgroups share an
// image); beyond that two or three contexts of eight work on an image each.
//
// What bounds it: at small batches the chain of latencies (frame loads, quantise, MMAs, requantise, three
// times over); at large ones the tensor pipe, which pays for 128 rows where the last two layers have 89
// and 61 (2 900 cycles an image against 2 300 with tiles that span images), and the issue of some 7 500
// warp instructions an image.  A whole step of the wide network, launched layer by layer / with this
// kernel: 26.4 / 15.5 us for 160 states (with the fc head), 43.5 / 42.2 for 1237; narrow 37.1 / 28.3 for 1237.
// (Three contexts need operands without padding rows and three accumulators in turns for the first layer;
// with two padded contexts 46.2 and 33.1.)
//
// Every wait is bounded.  A role whose wait gives up sets the status word and goes on (all further
// waits return at once).
#include <cuda.h>
#include <string.h>

#include "internal.h"
#include "tc_atari.h"
#include "tc_image.cuh"

namespace accerl {

namespace {

constexpr int kAtariCtx = 3;  // images in flight per CTA, at most

struct __align__(8) AtariBars {
    uint64_t w_ready;
    uint64_t ready[kAtariCtx][3];  // per context: the operand of layer l is complete
    uint64_t full1[kAtariCtx][4], empty1[kAtariCtx][4], full2[kAtariCtx], full3[kAtariCtx];  // accumulators
    uint32_t tmem_base;
    int abort_flag;
};

// byte offset of 16-byte piece `c` of row `row` of an operand with RB-byte rows under the RB-byte swizzle
template <int RB>
__device__ __forceinline__ uint32_t piece_off(int row, int c)
{
    if (RB == 128) return (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4));
    if (RB == 64) return (uint32_t)(row * 64 + ((c ^ ((row >> 1) & 3)) << 4));
    return (uint32_t)(row * 32 + ((c ^ ((row >> 2) & 1)) << 4));
}
template <int RB>
__host__ __device__ constexpr uint32_t rows_desc_hi()
{
    return (uint32_t)(8 * RB >> 4) | (1u << 14) | ((RB == 128 ? 2u : RB == 64 ? 4u : 6u) << 29);
}

// channels 16 * P .. 16 * P + 15 (the constants at addresses known at compile time)
template <int P>
__device__ __forceinline__ uint4 requant_piece(const int (&acc)[16], const AtariLayer &L)
{
    float ks[16], bs[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float4 kv = *reinterpret_cast<const float4 *>(&L.k[16 * P + 4 * g]);
        const float4 bv = *reinterpret_cast<const float4 *>(&L.b[16 * P + 4 * g]);
        ks[4 * g] = kv.x; ks[4 * g + 1] = kv.y; ks[4 * g + 2] = kv.z; ks[4 * g + 3] = kv.w;
        bs[4 * g] = bv.x; bs[4 * g + 1] = bv.y; bs[4 * g + 2] = bv.z; bs[4 * g + 3] = bv.w;
    }
    uint32_t w[4];
    if (L.affine) requant16_affine<false>(acc, ks, bs, w);
    else requant16_fastdiv<false>(acc, ks, bs, L.s_out, L.inv_s_out, w);
    const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
    return L.relu ? relu16(v) : v;
}

// F(OpIndex<p>) for the pieces p = wg, wg + WG, ... below N
template <int N, int WG, int P = 0, typename F>
__device__ __forceinline__ void for_pieces(int wg, F &&f)
{
    if constexpr (P < N) {
        if (P % WG == wg) f(OpIndex<P>());
        for_pieces<N, WG, P + 1>(wg, f);
    }
}

// four frame bytes -> four codes; MODE as in AtariParams
template <int MODE>
__device__ __forceinline__ uint32_t quantise_frame_word(uint32_t w, uint32_t mul, uint32_t add)
{
    if (MODE == 2) return (w >> 1) & 0x7f7f7f7fu;
    const uint32_t r0 = __byte_perm(w, 0, 0x4440) * mul + add, r1 = __byte_perm(w, 0, 0x4441) * mul + add;
    const uint32_t r2 = __byte_perm(w, 0, 0x4442) * mul + add, r3 = __byte_perm(w, 0, 0x4443) * mul + add;
    const uint32_t codes = __byte_perm(__byte_perm(r0, r1, 0x0073), __byte_perm(r2, r3, 0x0073), 0x5410);
    return MODE == 1 ? __vminu4(codes, 0x7f7f7f7fu) : codes;
}

constexpr int kb(int bytes) { return (bytes + 1023) & ~1023; }

// Memory of a network.  Shared: weights, then per context the three layers' operands, exactly as long as
// they are: the rows behind the last position that a tile and its taps touch are the next operand's (they
// only reach rows of the result that are no output), and a few rows of slack behind the last context.
// Tensor memory: four tiles of the first layer's accumulators (or three that take turns), and the columns
// that the second and the third layer share.
template <int C1, int C2, int C3, int CTX>
struct AtariSizes {
    static constexpr int w1 = 4 * C1 * 64, w2 = 4 * C2 * 4 * C1, w3 = 9 * C3 * C2, weights = w1 + w2 + w3;
    static constexpr int a1 = kb(441 * 64), a2 = kb(100 * 4 * C1), a3 = kb(81 * C2), ctx = a1 + a2 + a3;
    static constexpr int slack = 8 * 1024;
    static constexpr int slots = CTX * (4 * C1 + C2) <= 512 ? 4 : 3, col23 = slots * C1, cols = col23 + C2;
    static_assert(CTX <= kAtariCtx && CTX * cols <= 512 && 1024 + weights + CTX * ctx + slack <= 226 * 1024, "memory");
    static_assert(w1 % 1024 == 0 && w2 % 1024 == 0 && w3 % 1024 == 0 && C2 == C3, "swizzle atoms");
    // what the last context's operands reach beyond them
    static_assert((4 * 128 + 22) * 64 <= a1 + a2 + a3 + slack && (128 + 11) * 4 * C1 <= a2 + a3 + slack && (128 + 20) * C2 <= a3 + slack, "slack");
};

}  // namespace

template <int C1, int C2, int C3, int CTX, int WG, int MODE, bool TAP>
__global__ void __launch_bounds__(32 * (CTX * WG * 4 + CTX), 1) atari_kernel(const __grid_constant__ AtariParams p)
{
    using S = AtariSizes<C1, C2, C3, CTX>;
    // With three accumulators that take turns, tiles 0 and 3 of an image share one: whoever waits for tile 3
    // must have seen tile 0, or one behind it, complete; otherwise the wait's parity could mean the use before.
    static_assert(S::slots == 4 || WG <= 2, "a warpgroup that takes tile 3 only");
    constexpr int RB2 = 4 * C1, RB3 = C2, kEpi = CTX * WG * 4, kT = WG * 128;
    extern __shared__ __align__(1024) uint8_t atari_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)atari_smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ AtariBars bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int *abort_flag = &bars.abort_flag;

    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars.w_ready), 1);
        for (int c = 0; c < CTX; ++c) {
            for (int l = 0; l < 3; ++l) mbar_init(smem_u32(&bars.ready[c][l]), WG * 4);
            for (int t = 0; t < 4; ++t) {
                mbar_init(smem_u32(&bars.full1[c][t]), 1);
                mbar_init(smem_u32(&bars.empty1[c][t]), 4);
            }
            mbar_init(smem_u32(&bars.full2[c]), 1);
            mbar_init(smem_u32(&bars.full3[c]), 1);
        }
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async();
        mbar_expect_tx(smem_u32(&bars.w_ready), S::weights);
        bulk_load(smem_u32(smem), p.w, S::weights, smem_u32(&bars.w_ready));
    }
    if (warp == kEpi) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = bars.tmem_base;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int step = CTX * (int)gridDim.x, batch = routed_batch(p.route, p.batch);

    if (warp >= kEpi) {
        // ------------------------------------------------------------------ MMA issuers, one per context
        const int ctx = warp - kEpi;
        const uint32_t ready0 = smem_u32(&bars.ready[ctx][0]), full1 = smem_u32(&bars.full1[ctx][0]),
                       empty1 = smem_u32(&bars.empty1[ctx][0]);
        const uint32_t lo = 1u << 16, base = smem_u32(smem);
        const uint32_t b1 = (base >> 4) | lo, b2 = ((base + S::w1) >> 4) | lo, b3 = ((base + S::w1 + S::w2) >> 4) | lo;
        const uint32_t bufs = base + S::weights + (uint32_t)ctx * S::ctx;
        const uint32_t a1 = (bufs >> 4) | lo, a2 = ((bufs + S::a1) >> 4) | lo, a3 = ((bufs + S::a1 + S::a2) >> 4) | lo;
        const uint32_t d = tmem + (uint32_t)(ctx * S::cols), d23 = d + S::col23;
        uint32_t par1 = 0, par = 0, seq = 0;
        auto conv1 = [&]() {
            image_wait(ready0, par1, abort_flag, p.status, 8);
            par1 ^= 1;
            for (int t = 0; t < 4; ++t, ++seq) {
                const uint32_t slot = seq % S::slots;
                if (S::slots < 4) image_wait(empty1 + 8 * slot, ((seq / S::slots) & 1) ^ 1, abort_flag, p.status, 4);
                fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks)
                            mma_i8(d + slot * C1, desc(rows_desc_hi<64>(), a1 + (uint32_t)(t * 128 + (j >> 1) * 21 + (j & 1)) * 4 + 2 * ks),
                                   desc(rows_desc_hi<64>(), b1 + (uint32_t)(j * C1 * 4 + 2 * ks)), idesc_for(C1), (uint32_t)(j | ks));
                    mma_commit(full1 + 8 * slot);
                }
                __syncwarp();
            }
        };
        image_wait(smem_u32(&bars.w_ready), 0, abort_flag, p.status, 2);
        int n = (int)blockIdx.x + ctx * (int)gridDim.x;
        if (n < batch) conv1();
        for (; n < batch; n += step, par ^= 1) {
            image_wait(ready0 + 8, par, abort_flag, p.status, 8);
            fence_after();
            if (elect_one()) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int ks = 0; ks < RB2 / 32; ++ks)
                        mma_i8(d23, desc(rows_desc_hi<RB2>(), a2 + (uint32_t)((j >> 1) * 10 + (j & 1)) * (RB2 / 16) + 2 * ks),
                               desc(rows_desc_hi<RB2>(), b2 + (uint32_t)(j * C2 * (RB2 / 16) + 2 * ks)), idesc_for(C2), (uint32_t)(j | ks));
                mma_commit(smem_u32(&bars.full2[ctx]));
            }
            __syncwarp();
            image_wait(ready0 + 16, par, abort_flag, p.status, 8);
            fence_after();
            if (elect_one()) {
#pragma unroll
                for (int j = 0; j < 9; ++j)
#pragma unroll
                    for (int ks = 0; ks < RB3 / 32; ++ks)
                        mma_i8(d23, desc(rows_desc_hi<RB3>(), a3 + (uint32_t)((j / 3) * 9 + j % 3) * (RB3 / 16) + 2 * ks),
                               desc(rows_desc_hi<RB3>(), b3 + (uint32_t)(j * C3 * (RB3 / 16) + 2 * ks)), idesc_for(C3), (uint32_t)(j | ks));
                mma_commit(smem_u32(&bars.full3[ctx]));
            }
            __syncwarp();
            // the next image's first layer behind this image's third (in front of it, its fourth tile could wait
            // for an accumulator that is only read after the third layer)
            if (n + step < batch) conv1();
        }
    } else {
        // ------------------------------------------------------------------ frames in, accumulators out
        const int ctx = warp / (WG * 4), wg = (warp >> 2) % WG, q = warp & 3;
        const int tid = (int)threadIdx.x - ctx * kT, row = q * 32 + lane;
        const uint32_t a1 = smem_u32(smem) + S::weights + (uint32_t)ctx * S::ctx, a2 = a1 + S::a1, a3 = a2 + S::a2;
        const uint32_t ready0 = smem_u32(&bars.ready[ctx][0]), full1 = smem_u32(&bars.full1[ctx][0]),
                       empty1 = smem_u32(&bars.empty1[ctx][0]);
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ctx * S::cols);
        auto operand_done = [&](int layer) {  // this warp's share of it, and all its reads of accumulators before
            fence_async();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(ready0 + 8 * layer);
        };
        auto convert = [&](int n) {
            constexpr int kIter = (441 + kT - 1) / kT;
            const uint8_t *img = p.obs + (size_t)routed_row(p.route, n) * 28224;
            uint32_t w[kIter][16];
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = min(tid + j * kT, 440), Y = i / 21, X = i - Y * 21;
                const uint8_t *src = img + Y * 336 + X * 4;
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int dy = 0; dy < 4; ++dy) w[j][4 * c + dy] = __ldg(reinterpret_cast<const uint32_t *>(src + c * 7056 + dy * 84));
            }
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = tid + j * kT;
                if (i < 441)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        sts16(a1 + piece_off<64>(i, c), make_uint4(quantise_frame_word<MODE>(w[j][4 * c], p.ingest_mul, p.ingest_add),
                                                                   quantise_frame_word<MODE>(w[j][4 * c + 1], p.ingest_mul, p.ingest_add),
                                                                   quantise_frame_word<MODE>(w[j][4 * c + 2], p.ingest_mul, p.ingest_add),
                                                                   quantise_frame_word<MODE>(w[j][4 * c + 3], p.ingest_mul, p.ingest_add)));
            }
            operand_done(0);
            if (tid == 0 && n + step < batch)  // the image after this one on its way into L2
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.obs + (size_t)routed_row(p.route, n + step) * 28224), "r"(28224)
                             : "memory");
        };
        const int Y2 = row / 10, X2 = row - Y2 * 10, Y3 = row / 9, X3 = row - Y3 * 9;
        const bool v2 = Y2 < 9 && X2 < 9, v3 = Y3 < 7 && X3 < 7;
        int n = (int)blockIdx.x + ctx * (int)gridDim.x;
        if (n < batch) convert(n);
        uint32_t par = 0, seq0 = 0;
        for (; n < batch; n += step, par ^= 1, seq0 += 4) {
            // ---- first layer -> space-to-depth(2) rows
            for (int t = wg; t < 4; t += WG) {
                const int m = t * 128 + row, Y = m / 21, X = m - Y * 21;
                const bool v = Y < 20 && X < 20;
                const int r = (Y >> 1) * 10 + (X >> 1), at = ((Y & 1) * 2 + (X & 1)) * (C1 / 16);
                const uint32_t slot = (seq0 + t) % S::slots;
                image_wait(full1 + 8 * slot, ((seq0 + t) / S::slots) & 1, abort_flag, p.status, 16);
                fence_after();
                int a[C1 / 16][16];
#pragma unroll
                for (int i = 0; i < C1 / 16; ++i) tmem_ld16(tlane + slot * C1 + 16 * i, a[i]);
                tmem_wait_ld();
                if (S::slots < 4) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty1 + 8 * slot);
                }
                for_pieces<C1 / 16, 1>(0, [&](auto piece) {
                    constexpr int P = decltype(piece)::value;
                    const uint4 c = requant_piece<P>(a[P], p.layer[0]);
                    if (v) {
                        sts16(a2 + piece_off<RB2>(r, at + P), c);
                        if (TAP) *reinterpret_cast<uint4 *>(p.tap1 + ((size_t)n * 100 + r) * RB2 + (at + P) * 16) = c;
                    }
                });
            }
            operand_done(1);
            if (n + step < batch) {
                image_wait(full1 + 8 * ((seq0 + 3) % S::slots), ((seq0 + 3) / S::slots) & 1, abort_flag, p.status, 16);  // the last tile's MMAs have read the frame
                convert(n + step);
            }
            // ---- second layer
            image_wait(smem_u32(&bars.full2[ctx]), par, abort_flag, p.status, 16);
            fence_after();
            for_pieces<C2 / 16, WG>(wg, [&](auto piece) {
                constexpr int P = decltype(piece)::value;
                int a[16];
                tmem_ld16(tlane + S::col23 + 16 * P, a);
                tmem_wait_ld();
                const uint4 c = requant_piece<P>(a, p.layer[1]);
                if (v2) {
                    sts16(a3 + piece_off<RB3>(Y2 * 9 + X2, P), c);
                    if (TAP) *reinterpret_cast<uint4 *>(p.tap2 + ((size_t)n * 81 + Y2 * 9 + X2) * C2 + P * 16) = c;
                }
            });
            operand_done(2);
            // ---- third layer -> the fc layer's input rows
            image_wait(smem_u32(&bars.full3[ctx]), par, abort_flag, p.status, 16);
            fence_after();
            for_pieces<C3 / 16, WG>(wg, [&](auto piece) {
                constexpr int P = decltype(piece)::value;
                int a[16];
                tmem_ld16(tlane + S::col23 + 16 * P, a);
                tmem_wait_ld();
                const uint4 c = requant_piece<P>(a, p.layer[2]);
                if (v3) *reinterpret_cast<uint4 *>(p.out + ((size_t)n * 49 + Y3 * 7 + X3) * C3 + P * 16) = c;
            });
        }
    }

    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies in flight land
    fence_before();
    __syncthreads();
    if (warp == kEpi) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
template <int C1, int C2, int C3>
static cudaError_t atari_go(const AtariParams &p, int sm_count, cudaStream_t st)
{
    const int images = p.route.count ? p.route.expect : p.batch;
    auto go = [&](auto kernel, auto contexts, int wg) -> cudaError_t {
        constexpr int ctx = decltype(contexts)::value;
        using S = AtariSizes<C1, C2, C3, ctx>;
        const size_t smem = 1024 + S::weights + (size_t)ctx * S::ctx + S::slack;
        cudaError_t e = allow_smem((const void *)kernel, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(p.batch < sm_count ? p.batch : sm_count));
        cfg.blockDim = dim3((unsigned)(32 * (ctx * wg * 4 + ctx)));
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, p);
    };
    auto pick = [&](auto mode) -> cudaError_t {
        constexpr int M = decltype(mode)::value;
        if (p.tap1) return go(atari_kernel<C1, C2, C3, 1, 4, M, true>, OpIndex<1>(), 4);
        if (images <= sm_count) return go(atari_kernel<C1, C2, C3, 1, 4, M, false>, OpIndex<1>(), 4);
        // (the third context pays from three images per SM on: 160 states 15.5 against 16.5 us a step, 1237 states
        // 44.4 against 42.2, 32 / 64 / 64 channels)
        if (images <= 2 * sm_count) return go(atari_kernel<C1, C2, C3, 2, 2, M, false>, OpIndex<2>(), 2);
        return go(atari_kernel<C1, C2, C3, 3, 2, M, false>, OpIndex<3>(), 2);
    };
    return p.ingest_mode == 2 ? pick(OpIndex<2>()) : p.ingest_mode == 1 ? pick(OpIndex<1>()) : pick(OpIndex<0>());
}

cudaError_t atari_launch(const AtariParams &p, int sm_count, cudaStream_t st)
{
    return p.wide ? atari_go<32, 64, 64>(p, sm_count, st) : atari_go<16, 32, 32>(p, sm_count, st);
}

}  // namespace accerl
