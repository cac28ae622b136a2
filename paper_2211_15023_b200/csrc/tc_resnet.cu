// The IMPALA residual network with its images resident in shared memory: three launches from the
// frames to the fully connected layer's input.
//
//   res_first    frames -> quantise -> conv 3x3 (4 -> 16) at 84 x 84 -> max-pool        -> 41 x 41 x 16
//   res_stack1   two residual blocks at 41 x 41 -> conv 3x3 (16 -> 32) -> max-pool      -> 20 x 20 x 32
//   res_stack23  two blocks at 20 x 20 -> conv 3x3 -> max-pool -> two blocks at 9 x 9   -> 81 x 32
//
// Layer by layer (tc_mixed_plan.cu) every conv reads and writes its tensor, and often a second form
// of it, through HBM: 15 GB for 16384 states, 20 launches, 4.6 ms.  Here a CTA keeps an image's tensors
// in shared memory from one layer to the next, the tensor that a residual add needs in spare columns of
// tensor memory, and all weights of the kernel beside them; only the three tensors between the
// kernels touch HBM (74 KB a state with the frame).
//
// An image's layers depend on one another, so a CTA works on two or three images at once: contexts, each
// with its own issuing warp, warpgroups, buffers and part of tensor memory; while one context
// requantises, another's MMAs run.  Inside a context the 128-row tiles of a layer overlap as well:
// a tile is requantised while the next one is contracted.
//
// Convolutions are row-shifted implicit GEMMs as everywhere in this library: a GEMM row is 32 bytes of
// the stored image (two 16-channel pixels or one of 32 channels), a tap a fixed row offset.  16 channels:
// a row produces two output pixels (N = 2 * 16, banded weights, six K steps); 32 channels: one (N = 32,
// nine K steps).  N = 32 instructions cost 40 cycles, bound by reading their 4 KB operand: wider rows
// (N = 64, four pixels) would save a tenth of the tensor time and quadruple the weights' shared memory.
//
// A layer's operand is handed over tile by tile: a tile of the next layer is contracted as soon as the
// operand rows its taps reach are there (its own tile and the neighbours), so no layer ends in a wait for all
// of its warps; the issuing warp also lets the next image land as soon as its last MMA has read this one.
//
// What bounds it (counters at 4096 states, per image): the tensor pipe by instruction count (10 080 of 15 100 cycles
// in res_stack1, 8 640 of 12 800 in res_stack23; an MMA of N = 32 reads its operands at the full rate of shared
// memory) and instruction issue of the epilogues (35 300 and 24 100 warp instructions, 60 and 48 % of the slots; in
// res_stack1 about half of them convert and pack its 164 000 codes).
//
// Batch 16384, us per launch (with events between the launches; a step without them overlaps their ends) and step:
//   single-fma code in all three                          409 / 808 / 634   1861
//   the first layer divides, both sorts in the others     478 / 837 / 675   2002
//   every layer divides                                   476 / 908 / 706   2111
// One layer without single-fma constants gives its whole launch the code with both requantisers.  Of 60 drawn
// networks 6 have constants everywhere, of 20 calibrated ones none (first 13, stack 1 eight, stacks 2 and 3 none).
// Handed over by whole layers, both requantisers in all code: 489 / 841 / 769 for a policy that divides in the first
// layer and in some of stacks 2 and 3, as it is 478 / 810 / 674; 100 images of it, one context with two or four
// warpgroups: step 53.6 / 47.7.  A third warpgroup in res_first: 513 (spills) against its 478.
//
// Every wait is bounded.  A role whose wait gives up sets the status word and goes on (all further
// waits return at once), so that the barriers inside a context always see all their warps.
#include <cuda.h>
#include <string.h>

#include <type_traits>

#include "epilogue.cuh"
#include "internal.h"
#include "tc_image.cuh"
#include "tc_ptx.cuh"
#include "tc_resnet.h"

namespace accerl {

namespace {

constexpr int kMaxCtx = 3;  // images in flight per CTA
constexpr int kMaxSlots = 7;
constexpr int kMaxTiles = 7;  // 128-row tiles of a layer whose operand is waited for tile by tile


struct __align__(8) ResBars {
    uint64_t w_ready;
    uint64_t land[kMaxCtx];                // an image has arrived
    uint64_t ready[kMaxCtx][kMaxTiles];    // a tile of the next layer's operand (or all of it) is complete
    uint64_t acc_full[kMaxCtx][kMaxSlots], acc_empty[kMaxCtx][kMaxSlots];
    uint32_t tmem_base;
    int abort_flag;
};

// byte offset of 16-byte half `c` of 32-byte row `row` under the 32-byte swizzle
__device__ __forceinline__ uint32_t row_off(int row, int c) { return (uint32_t)(row * 32 + ((c ^ ((row >> 2) & 1)) << 4)); }

// all warps of a context's epilogue
template <int THREADS>
__device__ __forceinline__ void ctx_sync(int ctx)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + ctx), "n"(THREADS) : "memory");
}

// byte-wise maximum of signed bytes, two at a time as the high bytes of 16-bit lanes (the low bytes only
// decide between equal high bytes): `odd` keeps bytes 1 and 3 of the words seen, `even` bytes 0 and 2
struct ByteMax {
    uint32_t odd[4], even[4];
    __device__ __forceinline__ static uint32_t max2(uint32_t a, uint32_t b)
    {
        uint32_t r;
        asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    __device__ __forceinline__ void first(uint4 v)
    {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            odd[i] = w[i];
            even[i] = w[i] << 8;
        }
    }
    __device__ __forceinline__ void take(uint4 v)
    {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            odd[i] = max2(odd[i], w[i]);
            even[i] = max2(even[i], w[i] << 8);
        }
    }
    __device__ __forceinline__ uint4 result() const
    {
        return make_uint4(__byte_perm(even[0], odd[0], 0x7351), __byte_perm(even[1], odd[1], 0x7351),
                          __byte_perm(even[2], odd[2], 0x7351), __byte_perm(even[3], odd[3], 0x7351));
    }
};

// Sixteen accumulators of channels c0 .. c0 + 15 -> sixteen codes.  The constants are kernel parameters
// at addresses known at compile time (the layer loops are unrolled for that): indexed at run time they
// took the indexed-constant path (4 050 requests an image in res_stack23, half of that unit's peak, the
// contexts evicting each other's lines); from shared memory a broadcast 16-byte load costs four
// wavefronts of the port the MMAs read their operands through (res_stack1: 12 000 of 20 000 cycles an
// image); and held in registers over a layer they push the kernels into spills, which are deadly
// beside 220 KB of shared memory, with hardly any L1 left (2.4 ms instead of 1.1).
template <bool AFFINE, bool RELU>
__device__ __forceinline__ uint4 requant_res(const int (&acc)[16], const ResLayer &L, int c0)
{
    float ks[16], bs[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float4 kv = *reinterpret_cast<const float4 *>(&L.k[c0 + 4 * g]);
        const float4 bv = *reinterpret_cast<const float4 *>(&L.b[c0 + 4 * g]);
        ks[4 * g] = kv.x; ks[4 * g + 1] = kv.y; ks[4 * g + 2] = kv.z; ks[4 * g + 3] = kv.w;
        bs[4 * g] = bv.x; bs[4 * g + 1] = bv.y; bs[4 * g + 2] = bv.z; bs[4 * g + 3] = bv.w;
    }
    uint32_t w[4];
    if (AFFINE || L.affine) requant16_affine<RELU>(acc, ks, bs, w);
    else requant16_fastdiv<RELU>(acc, ks, bs, L.s_out, L.inv_s_out, w);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// acc[i] += skip_mul[c0 + i] * x[i], one dp2a each
__device__ __forceinline__ void add_skip(int (&acc)[16], uint4 x, const ResLayer &L, int c0)
{
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const uint4 m = *reinterpret_cast<const uint4 *>(&L.mul[c0 + 4 * g]);
        acc[4 * g] = __dp2a_lo((int)m.x, (int)w[g], acc[4 * g]);
        acc[4 * g + 1] = __dp2a_lo((int)m.y, (int)w[g], acc[4 * g + 1]);
        acc[4 * g + 2] = __dp2a_hi((int)m.z, (int)w[g], acc[4 * g + 2]);
        acc[4 * g + 3] = __dp2a_hi((int)m.w, (int)w[g], acc[4 * g + 3]);
    }
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ uint4 tmem_ld4(uint32_t taddr)
{
    uint4 v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(taddr) : "memory");
    return v;
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint4 v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// descriptors: constant upper words; the lower word is (address >> 4) | flags
constexpr uint32_t kDescSw32Hi = (256u >> 4) | (1u << 14) | (6u << 29);   // 32-byte rows, 32-byte swizzle
constexpr uint32_t kDescSw32Lo = 1u << 16;
constexpr uint32_t kDescFlatHi = (128u >> 4) | (1u << 14);                // 16-byte rows, no swizzle: 8-row groups 128 bytes apart,
constexpr uint32_t kDescFlatLo = (16u >> 4) << 16;                        // the second half of a K step is the next row
// what every kernel of this file does first: barriers, tensor memory, weights; returns the tensor-memory base
template <int EPI_WARPS>
__device__ __forceinline__ uint32_t res_setup(ResBars &bars, uint8_t *buffers, int buffer_bytes, uint8_t *w_smem,
                                              const uint8_t *w, uint32_t w_bytes, int warp, int epi_arrivals, int wide_slot,
                                              int tile_arrivals, int wide_ready)
{
    // borders and padding stay zero for the life of the CTA
    for (int i = threadIdx.x; i < buffer_bytes / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(buffers)[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars.w_ready), 1);
        for (int c = 0; c < kMaxCtx; ++c) {
            mbar_init(smem_u32(&bars.land[c]), 1);
            for (int t = 0; t < kMaxTiles; ++t) mbar_init(smem_u32(&bars.ready[c][t]), t == wide_ready ? epi_arrivals : tile_arrivals);
            for (int s = 0; s < kMaxSlots; ++s) {
                mbar_init(smem_u32(&bars.acc_full[c][s]), 1);
                mbar_init(smem_u32(&bars.acc_empty[c][s]), s == wide_slot ? epi_arrivals : 4);
            }
        }
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_async();
    if (warp == EPI_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x == 0) {
        mbar_expect_tx(smem_u32(&bars.w_ready), w_bytes);
        bulk_load(smem_u32(w_smem), w, w_bytes, smem_u32(&bars.w_ready));
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return bars.tmem_base;
}

__device__ __forceinline__ void res_teardown(ResBars &bars, int warp, int alloc_warp, uint32_t tmem_base)
{
    if (*(volatile int *)&bars.abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies in flight land
    fence_before();
    __syncthreads();
    if (warp == alloc_warp) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// frames -> first conv -> max-pool
// ---------------------------------------------------------------------------------------
// The quantised frame lies in shared memory as lines of 88 four-byte pixels, the image from pixel 4 and
// line 1 on.  A GEMM row starts every four pixels (16 bytes; unswizzled, so that the 32 bytes of a K
// step may overlap the next row's) and holds the eight pixels 4X - 4 .. 4X + 3 of a line: enough for
// the five outputs 4X - 2 .. 4X + 2 and thus for two pooled ones, whose three-pixel maxima are taken on
// the accumulators (the requantiser is non-decreasing): N = 5 * 16, one K step per tap row.  The
// maximum over three lines follows on the codes in shared memory.  The MMAs take 2 340 of an image's 7 750 cycles
// (4096 states), the 17 500 warp instructions 57 % of the issue slots; neither is full, as two images an SM take turns
// at two barriers a context.  55.8 k codes (83 lines of 42 pooled pixels) are requantised and stored before the second
// pass makes 26.9 k of them.
namespace {
constexpr int kFirstCtx = 2, kFirstWg = 2;                   // images in flight, warpgroups of each
constexpr int kFirstT = kFirstWg * 128, kFirstEpi = kFirstCtx * kFirstWg * 4;
constexpr int kFirstTiles = 15, kFirstSlots = 3;             // ceil(83 lines * 22 rows / 128)
constexpr int kFrameBytes = 31 * 1024, kHpBytes = 55 * 1024; // quantised frame (last tile reads past it), pooled lines
constexpr int kFirstSmem = 1024 + 8192 + kFirstCtx * (kFrameBytes + kHpBytes);
static_assert((kFirstTiles * 128 + 45) * 16 <= kFrameBytes && 83 * 21 * 32 <= kHpBytes, "buffers");
}  // namespace

template <bool SHIFT, bool TAP, bool AFFINE>
__global__ void __launch_bounds__(32 * (kFirstEpi + kFirstCtx), 1) res_first_kernel(const __grid_constant__ ResFirstParams p)
{
    extern __shared__ __align__(1024) uint8_t res_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)res_smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ ResBars bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *bufs = smem + 8192;
    const uint32_t tmem = res_setup<kFirstEpi>(bars, bufs, kFirstCtx * (kFrameBytes + kHpBytes), smem, p.w, kResFirstWeights,
                                               warp, kFirstWg * 4, -1, kFirstWg * 4, -1);
    volatile int *abort_flag = &bars.abort_flag;
    const int step = kFirstCtx * (int)gridDim.x, batch = routed_batch(p.route, p.batch);

    if (warp >= kFirstEpi) {
        // ------------------------------------------------------------------ MMA issuers
        const int ctx = warp - kFirstEpi;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]);
        const uint32_t a0 = ((smem_u32(bufs) + (uint32_t)ctx * (kFrameBytes + kHpBytes)) >> 4) | kDescFlatLo;
        const uint32_t b0 = (smem_u32(smem) >> 4) | kDescSw32Lo;
        image_wait(smem_u32(&bars.w_ready), 0, abort_flag, p.status, 2);
        uint32_t slot = 0, phase = 0, it = 0;
        for (int n = (int)blockIdx.x + ctx * (int)gridDim.x; n < batch; n += step, ++it) {
            image_wait(ready, it & 1, abort_flag, p.status, 8);
            fence_after();
            for (int t = 0; t < kFirstTiles; ++t) {
                image_wait(empty0 + 8 * slot, phase ^ 1, abort_flag, p.status, 4);
                fence_after();
                if (elect_one()) {
                    const uint32_t d = tmem + (uint32_t)ctx * 256 + slot * 80;
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky)
                        mma_i8(d, desc(kDescFlatHi, a0 + (uint32_t)(t * 128 + ky * 22)), desc(kDescSw32Hi, b0 + (uint32_t)(ky * 160)),
                               idesc_for(80), (uint32_t)ky);
                    mma_commit(full0 + 8 * slot);
                }
                __syncwarp();
                if (++slot == kFirstSlots) slot = 0, phase ^= 1;
            }
        }
    } else {
        // ------------------------------------------------------------------ conversion, epilogue, pool
        const int ctx = warp / (kFirstWg * 4), wg = (warp >> 2) % kFirstWg, q = warp & 3;
        const int tid = (int)threadIdx.x - ctx * kFirstT;
        const uint32_t frame = smem_u32(bufs) + (uint32_t)ctx * (kFrameBytes + kHpBytes), hp = frame + kFrameBytes;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]);
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)ctx * 256;
        auto convert = [&](int n) {
            constexpr int kGroups = 84 * 21, kIter = (kGroups + kFirstT - 1) / kFirstT;
            const uint32_t *src = reinterpret_cast<const uint32_t *>(p.obs + (size_t)routed_row(p.route, n) * 28224);
            uint32_t w[kIter][4];
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = tid + j * kFirstT;
                if (i < kGroups)
#pragma unroll
                    for (int c = 0; c < 4; ++c) w[j][c] = __ldg(src + c * 1764 + i);  // the planes' words in order
            }
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = tid + j * kFirstT;
                if (i < kGroups) {
                    const int y = i / 21, g = i - y * 21;
                    uint4 v;
                    if (SHIFT) v = ingest_shift_line16(w[j][0], w[j][1], w[j][2], w[j][3]);
                    else
                        v = make_uint4(ingest_fixed_line4<true>(w[j][0], w[j][1], w[j][2], w[j][3], 0, p.ingest_mul, p.ingest_add),
                                       ingest_fixed_line4<true>(w[j][0], w[j][1], w[j][2], w[j][3], 1, p.ingest_mul, p.ingest_add),
                                       ingest_fixed_line4<true>(w[j][0], w[j][1], w[j][2], w[j][3], 2, p.ingest_mul, p.ingest_add),
                                       ingest_fixed_line4<true>(w[j][0], w[j][1], w[j][2], w[j][3], 3, p.ingest_mul, p.ingest_add));
                    sts16(frame + (uint32_t)(((y + 1) * 22 + g + 1) * 16), v);
                    if (TAP) *reinterpret_cast<uint4 *>(p.tap_in + ((size_t)n * kGroups + i) * 16) = v;
                }
            }
            fence_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(ready);
            if (tid == 0 && n + step < batch)  // the image after this one on its way into L2
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.obs + (size_t)routed_row(p.route, n + step) * 28224), "r"(28224)
                             : "memory");
        };
        int n = (int)blockIdx.x + ctx * (int)gridDim.x;
        if (n < batch) convert(n);
        uint32_t seq0 = 0;  // accumulators handed over before this image
        for (; n < batch; n += step, seq0 += kFirstTiles) {
            for (int t = wg; t < kFirstTiles; t += kFirstWg) {
                const uint32_t seq = seq0 + (uint32_t)t, slot = seq % kFirstSlots;
                image_wait(full0 + 8 * slot, (seq / kFirstSlots) & 1, abort_flag, p.status, 16);
                fence_after();
                const int m = t * 128 + q * 32 + lane;
                const int y = m / 22, X = m - y * 22, R = y * 21 + X;
                const bool valid = X < 21 && y < 83;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int a[16], b[16];  // eight columns of the three pixels at a time
                    const uint32_t ta = tlane + slot * 80 + (uint32_t)(32 * j);
#pragma unroll
                    for (int h = 0; h < 16; h += 8) {
                        tmem_ld8(ta + h, a + h);
                        tmem_ld8(ta + h + 16, b);
                        tmem_ld8(ta + h + 32, b + 8);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) a[h + i] = __vimax3_s32(a[h + i], b[i], b[8 + i]);
                    }
                    if (j == 1) {
                        fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(empty0 + 8 * slot);
                    }
                    const uint4 v = requant_res<AFFINE, false>(a, p.layer, 0);
                    if (valid) sts16(hp + row_off(R, j), v);
                }
            }
            ctx_sync<kFirstT>(ctx);  // all lines pooled along x; the MMAs have read the frame
            if (n + step < batch) convert(n + step);
            int8_t *out = p.x1 + (size_t)n * kRes1Bytes;
            if (tid < 125) {  // the zero pixels: lines 0 and 42, the first one of the lines between
                const int s = tid < 42 ? tid : tid < 84 ? 42 * 42 + tid - 42 : (tid - 83) * 42;
                *reinterpret_cast<uint4 *>(out + row_off(s >> 1, s & 1)) = make_uint4(0, 0, 0, 0);
            }
            for (int i = tid; i < 41 * 41; i += kFirstT) {
                const int oy = i / 41, ox = i - oy * 41, s = ox + 1, R = 2 * oy * 21 + (s >> 1), c = s & 1;
                ByteMax mx;
                mx.first(lds16(hp + row_off(R, c)));
                mx.take(lds16(hp + row_off(R + 21, c)));
                mx.take(lds16(hp + row_off(R + 42, c)));
                const uint4 v = mx.result();
                *reinterpret_cast<uint4 *>(out + row_off((oy + 1) * 21 + (s >> 1), c)) = v;
                if (TAP) *reinterpret_cast<uint4 *>(p.tap_x1 + ((size_t)n * 1681 + i) * 16) = v;
            }
            ctx_sync<kFirstT>(ctx);  // before the next image's lines overwrite these
        }
    }
    res_teardown(bars, warp, kFirstEpi, tmem);
}

// ---------------------------------------------------------------------------------------
// two residual blocks at 41 x 41 x 16, conv 16 -> 32, max-pool
// ---------------------------------------------------------------------------------------
// Per context two buffers: the operand of a block's first conv (ReLU'd; the image lands there too) and
// the tensor between its two convs.  The block's input x, which the second conv adds, stays in tensor
// memory: the thread that adds it is the thread that wrote it.  The 16 -> 32 conv runs as two halves of
// sixteen output channels, so that the un-pooled half fits the buffer between the convs.
namespace {
constexpr int kS1Tiles = 7, kS1Ops = 6;                     // 41 * 21 GEMM rows; layers and half layers
constexpr int kS1Buf = 30 * 1024;                           // an image's rows and what the last tile reads past them
// CTX images in flight, WG warpgroups of each
template <int CTX, int WG>
struct S1Shape {
    static constexpr int T = WG * 128, Epi = CTX * WG * 4, Threads = 32 * (Epi + CTX);
    static constexpr int Slots = CTX == 1 ? kS1Tiles : 3;       // accumulators of a context
    static constexpr int XCol = Slots * 32, Cols = XCol + 8 * kS1Tiles;  // tensor memory: accumulators, then 8 columns of x per tile
    static constexpr int Smem = 1024 + kRes1Weights + CTX * 2 * kS1Buf;
    // Two warpgroups take the tiles of all layers in turn, so the odd seventh falls to one and the other
    // alternately; x's tiles (written in layers 1, read in 1 and 3) stay with one of them.  A warpgroup that
    // waits for an accumulator has seen one of the last `Slots` uses complete, so the wait's parity is
    // unambiguous; more warpgroups have an accumulator per tile and always the same tiles.
    __host__ __device__ static constexpr int shift(int op) { return WG == 2 && Slots < kS1Tiles ? op & 1 : 0; }
    static_assert((WG <= 2 || Slots == kS1Tiles) && Slots <= kMaxSlots && Cols * CTX <= 512, "tiles of a warpgroup");
};
static_assert((kS1Tiles * 128 + 2 * 21 + 1) * 32 <= kS1Buf && kS1Tiles <= kMaxTiles, "buffers");
}  // namespace

template <bool TAP, bool AFFINE, int CTX, int WG>
__global__ void __launch_bounds__(S1Shape<CTX, WG>::Threads, 1) res_stack1_kernel(const __grid_constant__ ResStack1Params p)
{
    using S = S1Shape<CTX, WG>;
    constexpr int kS1Ctx = CTX, kS1Wg = WG, kS1T = S::T, kS1Epi = S::Epi, kS1Slots = S::Slots, kS1XCol = S::XCol, kS1Cols = S::Cols;
    extern __shared__ __align__(1024) uint8_t res_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)res_smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ ResBars bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *bufs = smem + kRes1Weights;
    const uint32_t tmem = res_setup<kS1Epi>(bars, bufs, kS1Ctx * 2 * kS1Buf, smem, p.w, kRes1Weights, warp, kS1Wg * 4, -1, 4, -1);
    volatile int *abort_flag = &bars.abort_flag;
    const int step = kS1Ctx * (int)gridDim.x, batch = routed_batch(p.route, p.batch);

    if (warp >= kS1Epi) {
        // ------------------------------------------------------------------ MMA issuers
        const int ctx = warp - kS1Epi;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]);
        const uint32_t r0 = ((smem_u32(bufs) + (uint32_t)(ctx * 2) * kS1Buf) >> 4) | kDescSw32Lo, h0 = r0 + (kS1Buf >> 4);
        const uint32_t w0 = (smem_u32(smem) >> 4) | kDescSw32Lo;
        const uint32_t land_bar = smem_u32(&bars.land[ctx]);
        auto fetch = [&](int n) {
            if (elect_one()) {
                mbar_expect_tx(land_bar, kRes1Bytes);
                bulk_load((r0 & 0x3fff) << 4, p.x1 + (size_t)n * kRes1Bytes, kRes1Bytes, land_bar);
                if (n + step < batch)  // the image after this one on its way into L2
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.x1 + (size_t)(n + step) * kRes1Bytes), "r"(kRes1Bytes)
                                 : "memory");
            }
            __syncwarp();
        };
        int n = (int)blockIdx.x + ctx * (int)gridDim.x;
        if (n < batch) fetch(n);
        image_wait(smem_u32(&bars.w_ready), 0, abort_flag, p.status, 2);
        uint32_t slot = 0, phase = 0, rdy = 0;
        for (; n < batch; n += step) {
            for (int op = 0; op < kS1Ops; ++op) {
                const uint32_t a_op = (op == 1 || op == 3) ? h0 : r0, b_op = w0 + (uint32_t)op * (6 * 1024 >> 4);
                uint32_t last_full = 0, last_phase = 0;
                if (op < 5) image_wait(ready, rdy, abort_flag, p.status, 8);
                for (int t = 0; t < kS1Tiles; ++t) {
                    // a tile's taps reach 43 rows past it: it needs the operand tile after it too, not the whole layer
                    // (the second half of the last conv reads what the first half read)
                    if (op < 5 && t + 1 < kS1Tiles) image_wait(ready + 8 * (t + 1), rdy, abort_flag, p.status, 8);
                    image_wait(empty0 + 8 * slot, phase ^ 1, abort_flag, p.status, 4);
                    fence_after();
                    if (elect_one()) {
                        const uint32_t d = tmem + (uint32_t)ctx * kS1Cols + slot * 32, a = a_op + (uint32_t)t * (128 * 2);
#pragma unroll
                        for (int j = 0; j < 6; ++j)
                            mma_i8(d, desc(kDescSw32Hi, a + (uint32_t)((j >> 1) * 21 + (j & 1)) * 2), desc(kDescSw32Hi, b_op + (uint32_t)j * 64),
                                   idesc_for(32), (uint32_t)j);
                        mma_commit(full0 + 8 * slot);
                    }
                    __syncwarp();
                    last_full = full0 + 8 * slot;
                    last_phase = phase;
                    if (++slot == kS1Slots) slot = 0, phase ^= 1;
                }
                if (op < 5) rdy ^= 1;
                else if (n + step < batch) {  // the MMAs have read the image: the next one may land
                    image_wait(last_full, last_phase, abort_flag, p.status, 16);
                    fetch(n + step);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int ctx = warp / (kS1Wg * 4), wg = (warp >> 2) % kS1Wg, q = warp & 3;
        const int tid = (int)threadIdx.x - ctx * kS1T;
        const uint32_t rbuf = smem_u32(bufs) + (uint32_t)(ctx * 2) * kS1Buf, hbuf = rbuf + kS1Buf;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]), land_bar = smem_u32(&bars.land[ctx]);
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)ctx * kS1Cols;
        auto operand_done = [&](int t) {
            fence_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(ready + 8 * t);
        };
        auto first_tile = [&](int shift) { return (wg + shift) % kS1Wg; };
        // GEMM row m = 128 t + row of this thread: is its second pixel part of the image (bit t)?
        const int row = q * 32 + lane;
        uint32_t second = 0;
        for (int t = 0; t < kS1Tiles; ++t)
            if ((t * 128 + row) % 21 < 20 && t * 128 + row < 861) second |= 1u << t;
        uint32_t seq0 = 0, it = 0;  // tiles handed over before this layer, images
        for (int n = (int)blockIdx.x + ctx * (int)gridDim.x; n < batch; n += step, ++it) {
            // the image: x to tensor memory, ReLU(x) in place for the first conv
            image_wait(land_bar, it & 1, abort_flag, p.status, 1);
            for (int t = first_tile(S::shift(1)); t < kS1Tiles; t += kS1Wg) {
                const int m = t * 128 + row, r = m + 21;
                const bool v[2] = {m < 861, ((second >> t) & 1) != 0};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t at = rbuf + row_off(r + h, h ^ 1);
                    uint4 x = make_uint4(0, 0, 0, 0);
                    if (v[h]) {
                        x = lds16(at);
                        sts16(at, relu16(x));
                    }
                    tmem_st4(tlane + kS1XCol + 8 * t + 4 * h, x);
                }
                operand_done(t);
            }
            tmem_wait_st();
            auto layer = [&](auto op_c) {
                constexpr int op = decltype(op_c)::value, c0 = op == 5 ? 16 : 0;
                constexpr bool skip = op == 1 || op == 3;      // second conv of a block
                const ResLayer &L = p.layer[op < 4 ? op : 4];
                const uint32_t dst = skip ? rbuf : hbuf;
                for (int t = first_tile(S::shift(op)); t < kS1Tiles; t += kS1Wg) {
                    const uint32_t seq = seq0 + (uint32_t)t, slot = seq % kS1Slots;
                    const int m = t * 128 + row, r = m + 21;
                    const bool v[2] = {m < 861, ((second >> t) & 1) != 0};
                    image_wait(full0 + 8 * slot, (seq / kS1Slots) & 1, abort_flag, p.status, 16);
                    fence_after();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {  // the row's two pixels
                        int a[16];
                        tmem_ld16(tlane + slot * 32 + 16 * h, a);
                        uint4 x = make_uint4(0, 0, 0, 0);
                        if (skip) x = tmem_ld4(tlane + kS1XCol + 8 * t + 4 * h);
                        tmem_wait_ld();
                        if (h == 1) {
                            fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(empty0 + 8 * slot);
                        }
                        if (skip) add_skip(a, x, L, 0);
                        uint4 c = requant_res<AFFINE, op == 0 || op == 2>(a, L, c0);
                        if (TAP && op < 4 && v[h]) {
                            const int Y = m / 21, X = m - Y * 21;
                            *reinterpret_cast<uint4 *>(p.tap[op] + (((size_t)n * 41 + Y) * 41 + 2 * X + h) * 16) = c;
                        }
                        if (op == 1) {  // the next block's x; its first conv reads ReLU(x)
                            tmem_st4(tlane + kS1XCol + 8 * t + 4 * h, c);
                            c = relu16(c);
                        }
                        if (v[h]) sts16(dst + row_off(r + h, h ^ 1), c);
                    }
                    if (op < 4) operand_done(t);
                }
                seq0 += kS1Tiles;
                if (op == 1) tmem_wait_st();
                if (op < 4) return;
                // a half of the 16 -> 32 conv is complete: 3 x 3 stride-2 max over it
                ctx_sync<kS1T>(ctx);
                int8_t *out = p.x2 + (size_t)n * kRes2Bytes;
                if (tid < 62) {  // the zero pixels: lines 0 and 21, the first one of the lines between
                    const int s = tid < 21 ? tid : tid < 42 ? 21 * 21 + tid - 21 : (tid - 41) * 21;
                    *reinterpret_cast<uint4 *>(out + row_off(s, op - 4)) = make_uint4(0, 0, 0, 0);
                }
                for (int i = tid; i < 400; i += kS1T) {
                    const int oy = i / 20, ox = i - oy * 20, R = (2 * oy + 1) * 21 + ox;
                    ByteMax mx;
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const int rr = R + 21 * ky;
                        const uint4 u0 = lds16(hbuf + row_off(rr, 1)), u1 = lds16(hbuf + row_off(rr + 1, 0)),
                                    u2 = lds16(hbuf + row_off(rr + 1, 1));
                        if (ky == 0) mx.first(u0);
                        else mx.take(u0);
                        mx.take(u1);
                        mx.take(u2);
                    }
                    const uint4 c = mx.result();
                    *reinterpret_cast<uint4 *>(out + row_off((oy + 1) * 21 + ox + 1, op - 4)) = c;
                    if (TAP) *reinterpret_cast<uint4 *>(p.tap_x2 + ((size_t)n * 400 + i) * 32 + 16 * (op - 4)) = c;
                }
                ctx_sync<kS1T>(ctx);
            };
            layer(OpIndex<0>());
            layer(OpIndex<1>());
            layer(OpIndex<2>());
            layer(OpIndex<3>());
            layer(OpIndex<4>());
            layer(OpIndex<5>());
        }
    }
    res_teardown(bars, warp, kS1Epi, tmem);
}

// ---------------------------------------------------------------------------------------
// two residual blocks at 20 x 20 x 32, conv 32 -> 32, max-pool, two blocks at 9 x 9 x 32
// ---------------------------------------------------------------------------------------
// As above with one pixel per GEMM row.  At 9 x 9, where a layer is one tile, the two warpgroups of a
// context take half of the channels each and a thread keeps its part of x in registers.
namespace {
constexpr int kS2Tiles = 4, kS2Ops = 9;                     // 20 * 21 GEMM rows; layers
constexpr int kS2Buf = 18 * 1024, kS3Buf = 5 * 1024, kS2CtxBytes = 2 * kS2Buf + 2 * kS3Buf;
template <int CTX, int WG>
struct S2Shape {
    static constexpr int T = WG * 128, Epi = CTX * WG * 4, Threads = 32 * (Epi + CTX);
    static constexpr int Slots = CTX == 1 ? kS2Tiles : 3, Slot3 = Slots;     // accumulators of the tiles at 20 x 20, then one for the layers at 9 x 9
    static constexpr int XCol = (Slots + 1) * 32, Cols = XCol + 8 * kS2Tiles;  // x: 8 columns a tile behind them
    static constexpr int Smem = 1024 + kRes2Weights + CTX * kS2CtxBytes;
    static_assert((WG == 2 || (WG == kS2Tiles && Slots == kS2Tiles)) && Slots < kMaxSlots && Cols * CTX <= 512, "tiles of a warpgroup");
};
static_assert((kS2Tiles * 128 + 2 * 21 + 2) * 32 <= kS2Buf && (128 + 22) * 32 <= kS3Buf && kS2Tiles < kMaxTiles, "buffers");
}  // namespace

template <bool TAP, bool AFFINE, int CTX, int WG>
__global__ void __launch_bounds__(S2Shape<CTX, WG>::Threads, 1) res_stack23_kernel(const __grid_constant__ ResStack23Params p)
{
    using S = S2Shape<CTX, WG>;
    constexpr int kS2Ctx = CTX, kS2Wg = WG, kS2T = S::T, kS2Epi = S::Epi, kS2Slots = S::Slots, kS2Slot3 = S::Slot3, kS2XCol = S::XCol,
                  kS2Cols = S::Cols;
    extern __shared__ __align__(1024) uint8_t res_smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)res_smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ ResBars bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *bufs = smem + kRes2Weights;
    const uint32_t tmem = res_setup<kS2Epi>(bars, bufs, kS2Ctx * kS2CtxBytes, smem, p.w, kRes2Weights, warp, 8, kS2Slot3, 4,
                                            kS2Tiles);
    volatile int *abort_flag = &bars.abort_flag;
    const int step = kS2Ctx * (int)gridDim.x, batch = routed_batch(p.route, p.batch);

    if (warp >= kS2Epi) {
        // ------------------------------------------------------------------ MMA issuers
        const int ctx = warp - kS2Epi;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]);
        const uint32_t r0 = ((smem_u32(bufs) + (uint32_t)ctx * kS2CtxBytes) >> 4) | kDescSw32Lo, h0 = r0 + (kS2Buf >> 4),
                       r3 = h0 + (kS2Buf >> 4), h3 = r3 + (kS3Buf >> 4);
        const uint32_t w0 = (smem_u32(smem) >> 4) | kDescSw32Lo, d0 = tmem + (uint32_t)ctx * kS2Cols;
        const uint32_t land_bar = smem_u32(&bars.land[ctx]);
        auto fetch = [&](int n) {
            if (elect_one()) {
                mbar_expect_tx(land_bar, kRes2Bytes);
                bulk_load((r0 & 0x3fff) << 4, p.x2 + (size_t)n * kRes2Bytes, kRes2Bytes, land_bar);
                if (n + step < batch)  // the image after this one on its way into L2
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.x2 + (size_t)(n + step) * kRes2Bytes), "r"(kRes2Bytes)
                                 : "memory");
            }
            __syncwarp();
        };
        int n = (int)blockIdx.x + ctx * (int)gridDim.x;
        if (n < batch) fetch(n);
        image_wait(smem_u32(&bars.w_ready), 0, abort_flag, p.status, 2);
        uint32_t rdy = 0, slot = 0, phase = 0, k3 = 0;  // k3: layers done at 9 x 9
        for (; n < batch; n += step) {
            for (int op = 0; op < kS2Ops; ++op) {
                const uint32_t b_op = w0 + (uint32_t)op * (9 * 1024 >> 4);
                if (op < 5) {
                    const uint32_t a_op = (op == 1 || op == 3) ? h0 : r0;
                    uint32_t last_full = 0, last_phase = 0;
                    image_wait(ready, rdy, abort_flag, p.status, 8);
                    for (int t = 0; t < kS2Tiles; ++t) {
                        // a tile's taps reach 44 rows past it: it needs the operand tile after it too, not the whole layer
                        if (t + 1 < kS2Tiles) image_wait(ready + 8 * (t + 1), rdy, abort_flag, p.status, 8);
                        image_wait(empty0 + 8 * slot, phase ^ 1, abort_flag, p.status, 4);
                        fence_after();
                        if (elect_one()) {
                            const uint32_t a = a_op + (uint32_t)t * (128 * 2);
#pragma unroll
                            for (int j = 0; j < 9; ++j)
                                mma_i8(d0 + slot * 32, desc(kDescSw32Hi, a + (uint32_t)((j / 3) * 21 + j % 3) * 2),
                                       desc(kDescSw32Hi, b_op + (uint32_t)j * 64), idesc_for(32), (uint32_t)j);
                            mma_commit(full0 + 8 * slot);
                        }
                        __syncwarp();
                        last_full = full0 + 8 * slot;
                        last_phase = phase;
                        if (++slot == kS2Slots) slot = 0, phase ^= 1;
                    }
                    rdy ^= 1;
                    if (op == 4 && n + step < batch) {  // the MMAs have read the image: the next one may land
                        image_wait(last_full, last_phase, abort_flag, p.status, 16);
                        fetch(n + step);
                    }
                } else {
                    const uint32_t a_op = (op == 6 || op == 8) ? h3 : r3;
                    image_wait(ready + 8 * kS2Tiles, k3 & 1, abort_flag, p.status, 8);
                    image_wait(empty0 + 8 * kS2Slot3, (k3 & 1) ^ 1, abort_flag, p.status, 4);
                    fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int j = 0; j < 9; ++j)
                            mma_i8(d0 + kS2Slot3 * 32, desc(kDescSw32Hi, a_op + (uint32_t)((j / 3) * 10 + j % 3) * 2),
                                   desc(kDescSw32Hi, b_op + (uint32_t)j * 64), idesc_for(32), (uint32_t)j);
                        mma_commit(full0 + 8 * kS2Slot3);
                    }
                    __syncwarp();
                    ++k3;
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int ctx = warp / (kS2Wg * 4), wg = (warp >> 2) % kS2Wg, q = warp & 3;
        const uint32_t rbuf = smem_u32(bufs) + (uint32_t)ctx * kS2CtxBytes, hbuf = rbuf + kS2Buf, r3buf = hbuf + kS2Buf,
                       h3buf = r3buf + kS3Buf;
        const uint32_t ready = smem_u32(&bars.ready[ctx][0]), full0 = smem_u32(&bars.acc_full[ctx][0]),
                       empty0 = smem_u32(&bars.acc_empty[ctx][0]), land_bar = smem_u32(&bars.land[ctx]);
        const uint32_t tctx = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ctx * kS2Cols);
        auto operand_done = [&](int t) {  // tile t at 20 x 20, or (kS2Tiles) a warp's part at 9 x 9
            fence_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(ready + 8 * t);
        };
        const int row = q * 32 + lane;
        uint32_t inside = 0;  // bit t: row 128 t + row is a pixel of the 20 x 20 image
        for (int t = 0; t < kS2Tiles; ++t)
            if ((t * 128 + row) % 21 < 20 && t * 128 + row < 420) inside |= 1u << t;
        const uint32_t off2 = row_off(row + 22, 0);  // first half of the row of tile 0; the other half: ^ 16, tile t: + 4096 t
        const int Y3 = row / 10, X3 = row - Y3 * 10;
        const bool v3 = Y3 < 9 && X3 < 9;
        const uint32_t off3 = row_off(row + 11, wg);
        uint32_t seq0 = 0, k3 = 0, it = 0;
        for (int n = (int)blockIdx.x + ctx * (int)gridDim.x; n < batch; n += step, ++it) {
            image_wait(land_bar, it & 1, abort_flag, p.status, 1);
            for (int t = wg; t < kS2Tiles; t += kS2Wg) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t at = rbuf + (off2 ^ (16 * h)) + t * 4096;
                    uint4 x = make_uint4(0, 0, 0, 0);
                    if ((inside >> t) & 1) {
                        x = lds16(at);
                        sts16(at, relu16(x));
                    }
                    tmem_st4(tctx + kS2XCol + 8 * t + 4 * h, x);
                }
                operand_done(t);
            }
            tmem_wait_st();
            auto layer20 = [&](auto op_c) {
                constexpr int op = decltype(op_c)::value;
                constexpr bool skip = op == 1 || op == 3;
                const ResLayer &L = p.layer[op];
                const uint32_t dst = skip ? rbuf : hbuf;
                for (int t = wg; t < kS2Tiles; t += kS2Wg) {
                    const uint32_t seq = seq0 + (uint32_t)t, slot = seq % kS2Slots;
                    const bool v = (inside >> t) & 1;
                    image_wait(full0 + 8 * slot, (seq / kS2Slots) & 1, abort_flag, p.status, 16);
                    fence_after();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        int a[16];
                        uint4 x = make_uint4(0, 0, 0, 0);
                        tmem_ld16(tctx + slot * 32 + 16 * h, a);
                        if (skip) x = tmem_ld4(tctx + kS2XCol + 8 * t + 4 * h);
                        tmem_wait_ld();
                        if (h == 1) {
                            fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(empty0 + 8 * slot);
                        }
                        if (skip) add_skip(a, x, L, 16 * h);
                        uint4 c = requant_res<AFFINE, op == 0 || op == 2>(a, L, 16 * h);
                        if (TAP && v) {
                            const int m = t * 128 + row, Y = m / 21, X = m - Y * 21;
                            *reinterpret_cast<uint4 *>(p.tap[op] + (((size_t)n * 20 + Y) * 20 + X) * 32 + 16 * h) = c;
                        }
                        if (op == 1) {  // the next block's x; its first conv reads ReLU(x)
                            tmem_st4(tctx + kS2XCol + 8 * t + 4 * h, c);
                            c = relu16(c);
                        }
                        if (v) sts16(dst + (off2 ^ (16 * h)) + t * 4096, c);
                    }
                    if (op < 4) operand_done(t);
                }
                seq0 += kS2Tiles;
                if (op == 1) tmem_wait_st();
            };
            layer20(OpIndex<0>());
            layer20(OpIndex<1>());
            layer20(OpIndex<2>());
            layer20(OpIndex<3>());
            layer20(OpIndex<4>());
            // 3 x 3 stride-2 max over the last one: every thread its pixel and channels of the 9 x 9 tensor
            ctx_sync<kS2T>(ctx);
            if (wg >= 2) continue;  // (two warpgroups do the layers at 9 x 9)
            uint4 x = make_uint4(0, 0, 0, 0);
            if (v3) {
                const int R = (2 * Y3 + 1) * 21 + 2 * X3 + 1;
                ByteMax mx;
                mx.first(lds16(hbuf + row_off(R, wg)));
#pragma unroll
                for (int j = 1; j < 9; ++j) mx.take(lds16(hbuf + row_off(R + (j / 3) * 21 + j % 3, wg)));
                x = mx.result();
                sts16(r3buf + off3, relu16(x));
                if (TAP) *reinterpret_cast<uint4 *>(p.tap_x3 + (((size_t)n * 9 + Y3) * 9 + X3) * 32 + 16 * wg) = x;
            }
            operand_done(kS2Tiles);
            auto layer9 = [&](auto op_c, auto half_c) {
                constexpr int op = decltype(op_c)::value, half = decltype(half_c)::value;
                constexpr bool skip = op == 6 || op == 8;
                const ResLayer &L = p.layer[op];
                image_wait(full0 + 8 * kS2Slot3, k3 & 1, abort_flag, p.status, 16);
                fence_after();
                int a[16];
                tmem_ld16(tctx + kS2Slot3 * 32 + 16 * half, a);
                tmem_wait_ld();
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8 * kS2Slot3);
                if (skip) add_skip(a, x, L, 16 * half);
                uint4 c = requant_res<AFFINE, op == 5 || op == 7>(a, L, 16 * half);
                if (TAP && v3 && op < 8) *reinterpret_cast<uint4 *>(p.tap[op] + (((size_t)n * 9 + Y3) * 9 + X3) * 32 + 16 * half) = c;
                if (skip) {
                    x = c;
                    c = relu16(c);
                }
                if (op == 8) {
                    if (v3) *reinterpret_cast<uint4 *>(p.x3 + (size_t)n * kRes3Bytes + (Y3 * 9 + X3) * 32 + 16 * half) = c;
                } else {
                    if (v3) sts16((skip ? r3buf : h3buf) + off3, c);
                    operand_done(kS2Tiles);
                }
                ++k3;
            };
            auto layers9 = [&](auto half_c) {
                layer9(OpIndex<5>(), half_c);
                layer9(OpIndex<6>(), half_c);
                layer9(OpIndex<7>(), half_c);
                layer9(OpIndex<8>(), half_c);
            };
            if (wg == 0) layers9(OpIndex<0>());
            else layers9(OpIndex<1>());
        }
    }
    res_teardown(bars, warp, kS2Epi, tmem);
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
namespace {

template <typename K, typename P>
cudaError_t res_launch(K kernel, const P &p, int threads, size_t smem, int sm_count, cudaStream_t st)
{
    cudaError_t e = allow_smem((const void *)kernel, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    // context c of CTA i starts with image i + c * CTAs: the second contexts come into play when every SM has an image
    cfg.gridDim = dim3((unsigned)(p.batch < sm_count ? p.batch : sm_count));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace

// Calls `go(TAP, AFFINE)` with both as compile-time values.  Kernels whose layers all have the single-fma pair do
// without the division's code (half of the requantiser's instructions, and the unrolled layers exceed the
// instruction cache), with and without parity taps.
template <typename F>
cudaError_t res_dispatch(const ResLayer *layer, int layers, bool tap, F go)
{
    bool affine = true;
    for (int i = 0; i < layers; ++i) affine &= layer[i].affine != 0;
    if (tap) return affine ? go(std::true_type(), std::true_type()) : go(std::true_type(), std::false_type());
    return affine ? go(std::false_type(), std::true_type()) : go(std::false_type(), std::false_type());
}

cudaError_t res_first_launch(const ResFirstParams &p, int sm_count, cudaStream_t st)
{
    return res_dispatch(&p.layer, 1, p.tap_in != nullptr, [&](auto tap, auto affine) {
        auto go = [&](auto kernel) { return res_launch(kernel, p, 32 * (kFirstEpi + kFirstCtx), kFirstSmem, sm_count, st); };
        return p.ingest_mode == 2 ? go(res_first_kernel<true, tap(), affine()>) : go(res_first_kernel<false, tap(), affine()>);
    });
}

// Up to an image per SM only one context would work: then it has all the warps (four warpgroups).
cudaError_t res_stack1_launch(const ResStack1Params &p, int sm_count, cudaStream_t st)
{
    return res_dispatch(p.layer, 5, p.tap_x2 != nullptr, [&](auto tap, auto affine) {
        if (p.batch <= sm_count)
            return res_launch(res_stack1_kernel<tap(), affine(), 1, 4>, p, S1Shape<1, 4>::Threads, S1Shape<1, 4>::Smem, sm_count, st);
        return res_launch(res_stack1_kernel<tap(), affine(), 3, 2>, p, S1Shape<3, 2>::Threads, S1Shape<3, 2>::Smem, sm_count, st);
    });
}

cudaError_t res_stack23_launch(const ResStack23Params &p, int sm_count, cudaStream_t st)
{
    return res_dispatch(p.layer, 9, p.tap_x3 != nullptr, [&](auto tap, auto affine) {
        if (p.batch <= sm_count)
            return res_launch(res_stack23_kernel<tap(), affine(), 1, 4>, p, S2Shape<1, 4>::Threads, S2Shape<1, 4>::Smem, sm_count, st);
        return res_launch(res_stack23_kernel<tap(), affine(), 3, 2>, p, S2Shape<3, 2>::Threads, S2Shape<3, 2>::Smem, sm_count, st);
    });
}

}  // namespace accerl
