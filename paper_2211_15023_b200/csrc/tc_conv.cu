// Strided, unpadded convolutions on int8 activations (the second and third layer of the paper's
// Atari networks, table "network architecture and inference time"): a conv with stride s and window
// k = s * t on a tensor stored space-to-depth(s) is a t x t stride-1 conv on its grid.
//
// A tile is ONE grid line of G = 128 / grid_w images (12 x 10 or 14 x 9 positions for the Atari layers): its
// 128 GEMM rows are (image, x).  So the operand tile of input line y has the same rows as the accumulators of
// the output lines y, y - 1, .. y - t + 1 it contributes to, one per vertical tap, and ONE instruction serves
// all of them: N = t * 64, the weights of the vertical taps side by side and the accumulators of t consecutive
// lines in consecutive columns of tensor memory.  An instruction costs max(39, 32 + N / 4, N / 2) cycles, so
// t of them at N = 64 (48 each) become one at 64 (t = 2) or 96 (t = 3).  Tiles of whole grid rows with a
// row-shifted operand per tap, as the other kernels have them, took 640 and 555 cycles an image for the
// second and third layer, these take 430 and 310.  (The first instruction on a new line must overwrite it
// and not the lines beside it, and lines that wrap around the ring of accumulators are two pieces: a few
// per cent.)  Horizontal taps are row-shifted views of the tile.
//
// - A pipeline stage is one input line: one four-dimensional TMA box (row bytes, x, one y, G images).
// - The CTAs share the (group of images, output line) pairs evenly; a CTA's range starts and ends anywhere in a
//   group and costs the t - 1 input lines before its first output line.
// - Scales and biases are kernel parameters read from the constant bank, because shared-memory loads of the
//   epilogue queue behind the operand reads of the MMAs.
//
// Every wait is bounded; a wait that gives up sets the status word and all roles leave.
#include <cuda.h>

#include <algorithm>

#include "epilogue.cuh"
#include "internal.h"
#include "tc_conv.h"
#include "tc_ptx.cuh"

namespace accerl {

namespace {

constexpr int kEpiWarps2 = 16;           // warps 0..15 drain accumulators
constexpr int kMmaWarp2 = kEpiWarps2, kTmaWarp2 = kEpiWarps2 + 1;
constexpr int kThreads2 = 32 * (kEpiWarps2 + 2);
constexpr int kMaxStages2 = 12, kMaxSlots2 = 16;

struct __align__(8) Bars2 {
    uint64_t full[kMaxStages2], empty[kMaxStages2];
    uint64_t acc_full[kMaxSlots2], acc_empty[kMaxSlots2];
    uint64_t b_ready;
    uint32_t tmem_base;
    int abort_flag;
};

// the single warps that issue and load wait without sleeping first: the whole CTA waits for them
__device__ __forceinline__ bool line_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    return mbar_wait_limited(bar, parity, abort_flag, status, code, 2048, kWaitLimitPolls);
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

}  // namespace

template <int NCOLS, bool AFFINE>
__global__ void __launch_bounds__(kThreads2, 1)
conv_rows_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                 const __grid_constant__ ConvRowsParams p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw2[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw2 + 1023) & ~(uintptr_t)1023);
    __shared__ Bars2 bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kAccSlots = 512 / NCOLS < kMaxSlots2 ? 512 / NCOLS : kMaxSlots2;  // ring of accumulators, NCOLS columns each
    const int RB = p.row_bytes, taps = p.taps;
    const int b_bytes = taps * taps * NCOLS * RB;
    uint8_t *b_tiles = smem;
    uint8_t *stages = smem + ((b_bytes + 1023) & ~1023);
    const int n_stages = p.n_stages;
    volatile int *abort_flag = &bars.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 1);
            mbar_init(smem_u32(&bars.empty[s]), 1);
        }
        for (int a = 0; a < kAccSlots; ++a) {
            mbar_init(smem_u32(&bars.acc_full[a]), 1);
            mbar_init(smem_u32(&bars.acc_empty[a]), 4);
        }
        mbar_init(smem_u32(&bars.b_ready), 1);
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kMmaWarp2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&bars.tmem_base)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = bars.tmem_base;
    // the next launch may set itself up while this grid drains
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // this CTA's output lines, numbered through all groups of images
    const int out_h = p.out_h;
    const int line0 = (int)((long long)blockIdx.x * p.total_lines / gridDim.x);
    const int n_lines = (int)((long long)(blockIdx.x + 1) * p.total_lines / gridDim.x) - line0;
    const int group0 = line0 / out_h, y0 = line0 - group0 * out_h;
    const uint32_t full0 = smem_u32(&bars.full[0]), empty0 = smem_u32(&bars.empty[0]);
    const uint32_t acc_full0 = smem_u32(&bars.acc_full[0]), acc_empty0 = smem_u32(&bars.acc_empty[0]);

    if (warp == kMmaWarp2) {
        // ------------------------------------------------------------------ MMA issuer
        const int ksteps = RB >> 5, n_j = taps * ksteps;  // 32-byte K steps of a position, of all horizontal taps
        if (elect_one()) {  // weights: per K step the vertical taps side by side, the last one first, in rows of 32 bytes
            mbar_expect_tx(smem_u32(&bars.b_ready), (uint32_t)b_bytes);
            for (int j = 0; j < n_j; ++j)
                for (int b = 0; b < taps; ++b)
                    tma_load_2d(smem_u32(b_tiles) + (j * taps + b) * NCOLS * 32, &map_b, 32 * (j % ksteps),
                                ((taps - 1 - b) * taps + j / ksteps) * NCOLS, smem_u32(&bars.b_ready));
        }
        __syncwarp();
        bool ok = mbar_wait(smem_u32(&bars.b_ready), 0, abort_flag, p.status, 2);
        auto idesc = [](int lines) {
            return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(lines * (NCOLS >> 3)) << 17) | ((uint32_t)(128 >> 4) << 24);
        };
        // descriptors: constant upper word | (address >> 4); operand rows of RB bytes, weights of 32, swizzled K-major
        const uint64_t a_hi = (uint64_t)(((uint32_t)(8 * RB) >> 4) | (1u << 14) | ((RB == 128 ? 2u : (RB == 64 ? 4u : 6u)) << 29)) << 32;
        const uint64_t b_hi = (uint64_t)((256u >> 4) | (1u << 14) | (6u << 29)) << 32;
        const uint32_t lo_flags = 1u << 16;
        const uint32_t b_lo = (smem_u32(b_tiles) >> 4) | lo_flags, a_lo = (smem_u32(stages) >> 4) | lo_flags;
        constexpr uint32_t b_line = NCOLS * 32 / 16;
        const uint32_t b_step = (uint32_t)taps * b_line, stage16 = (uint32_t)(p.stage_bytes >> 4);
        int stage = 0;
        uint32_t phase = 0, a0 = a_lo;
        int slot = 0;            // accumulator of the lowest line that is still being added to
        int new_slot = 0;        // and of the next new line
        uint32_t new_phase = 1;
        int ya = y0, left = n_lines;
        while (left > 0 && ok) {  // a segment: output lines ya .. yb - 1 of one group
            const int yb = min(out_h, ya + left);
            for (int y = ya; y < yb + taps - 1; ++y) {
                const int lo = max(ya, y - taps + 1), lines = min(yb - 1, y) - lo + 1;  // output lines lo .. lo + lines - 1
                const bool fresh = y < yb;                                              // the last of them is new
                const uint32_t d_new = tmem_base + (uint32_t)(new_slot * NCOLS);
                if (fresh) {
                    ok = line_wait(acc_empty0 + 8 * new_slot, new_phase, abort_flag, p.status, 4);
                    if (!ok) break;
                    if (++new_slot == kAccSlots) new_slot = 0, new_phase ^= 1;
                }
                ok = line_wait(full0 + 8 * stage, phase, abort_flag, p.status, 8);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const bool complete = y - taps + 1 >= ya;  // the lowest line is complete with this one
                if (elect_one()) {
                    // Lines in consecutive columns: n1 of them, and n2 that wrap around the ring.  A short loop and not
                    // straight-line code: the warp shares its scheduler's instruction buffer with the epilogue's long
                    // code and executes nothing that is not in a loop from there.
                    const int n1 = min(lines, kAccSlots - slot), n2 = lines - n1;
                    const uint32_t d1 = tmem_base + (uint32_t)(slot * NCOLS), i1 = idesc(n1), i2 = idesc(n2);
                    uint64_t a = a_hi | a0, b1 = b_hi | (b_lo + (uint32_t)(taps - 1 - (y - lo)) * b_line);
                    const uint64_t b12 = (uint64_t)((uint32_t)n1 * b_line);
                    int j = 0;
                    if (fresh) {  // the first instruction on a new line overwrites it
                        const int old = lines - 1, o1 = min(old, n1), o2 = old - o1;
                        mma_i8(d_new, a, b1 + (uint32_t)old * b_line, idesc(1), 0);
                        if (o1) mma_i8(d1, a, b1, idesc(o1), 1);
                        if (o2) mma_i8(tmem_base, a, b1 + b12, idesc(o2), 1);
                        j = 1;
                        a += 2;
                        b1 += b_step;
                    }
#pragma unroll 1
                    for (; j < n_j; ++j) {
                        mma_i8(d1, a, b1, i1, 1);
                        if (n2) mma_i8(tmem_base, a, b1 + b12, i2, 1);
                        a += 2;  // the horizontal taps and their K steps are consecutive 32-byte pieces
                        b1 += b_step;
                    }
                    mma_commit(empty0 + 8 * stage);  // the stage is free when these MMAs retire
                    if (complete) mma_commit(acc_full0 + 8 * slot);
                }
                __syncwarp();
                if (complete && ++slot == kAccSlots) slot = 0;
                a0 += stage16;
                if (++stage == n_stages) stage = 0, phase ^= 1, a0 = a_lo;
            }
            left -= yb - ya;
            ya = 0;
        }
    } else if (warp == kTmaWarp2) {
        // ------------------------------------------------------------------ TMA producer
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the activations are the previous launch's output
        bool ok = true;
        int stage = 0, ya = y0, left = n_lines, image = group0 * p.images;
        uint32_t phase = 0;
        const uint32_t bytes = (uint32_t)(p.images * p.grid_w * RB);
        while (left > 0 && ok) {
            const int yb = min(out_h, ya + left);
            for (int y = ya; y < yb + taps - 1; ++y) {
                ok = line_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, p.status, 1);
                if (!ok) break;
                if (elect_one()) {
                    mbar_expect_tx(full0 + 8 * stage, bytes);
                    tma_load_4d(smem_u32(stages) + (uint32_t)(stage * p.stage_bytes), &map_a, 0, 0, y, image, full0 + 8 * stage);
                }
                __syncwarp();
                if (++stage == n_stages) stage = 0, phase ^= 1;
            }
            left -= yb - ya;
            ya = 0;
            image += p.images;
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int wg = warp >> 2, q = warp & 3;
        constexpr int kGroups = kEpiWarps2 / 4;
        const int r = q * 32 + lane;  // this thread's row of every tile: position X of image `in_group` of the group
        const int in_group = r / p.grid_w, X = r - in_group * p.grid_w;
        const int sh = p.out_s2d_log2, smask = (1 << sh) - 1;
        const bool row_ok = in_group < p.images && X < p.out_w;
        const int x_off = (X >> sh) * p.out_pitch + (X & smask) * p.n_total;
        const float s_out = p.s_out, inv_s_out = p.inv_s_out;
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the output may reuse a buffer an earlier launch reads
        bool ok = true;
        int Y = y0 + wg, group = group0;
        for (int seq = wg; seq < n_lines && ok; seq += kGroups, Y += kGroups) {  // every fourth line of the CTA
            while (Y >= out_h) Y -= out_h, ++group;
            const int slot = seq % kAccSlots;
            ok = mbar_wait(acc_full0 + 8 * slot, (uint32_t)((seq / kAccSlots) & 1), abort_flag, p.status, 16);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(slot * NCOLS);
            const int n = group * p.images + in_group;
            const bool valid = row_ok && n < p.batch;
            int8_t *dst = p.out + (size_t)((unsigned)n * (unsigned)p.out_rows_per_image + (unsigned)((Y >> sh) * p.out_grid_w)) *
                                      (size_t)p.out_pitch +
                          (((Y & smask) << sh) * p.n_total + x_off);
            constexpr int kHalves = (NCOLS + 31) / 32;  // 32 columns at a time
#pragma unroll
            for (int hh = 0; hh < kHalves; ++hh) {
                constexpr int kPieces = NCOLS >= 32 ? 2 : 1;
                int acc[kPieces][16];
#pragma unroll
                for (int h = 0; h < kPieces; ++h) tmem_ld16(taddr + 32 * hh + 16 * h, acc[h]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (hh == kHalves - 1) {  // the last read of the accumulator: hand it back
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_empty0 + 8 * slot);
                }
                uint32_t wq[kPieces][4];
#pragma unroll
                for (int h = 0; h < kPieces; ++h) {
                    if (32 * hh + 16 * h >= NCOLS) continue;
                    float ks[16], bs[16];
#pragma unroll
                    for (int g = 0; g < 4; ++g) {  // kernel parameters: 16-byte reads from the constant bank
                        const float4 kv = *reinterpret_cast<const float4 *>(&p.ks[32 * hh + 16 * h + 4 * g]);
                        const float4 bv = *reinterpret_cast<const float4 *>(&p.bs[32 * hh + 16 * h + 4 * g]);
                        ks[4 * g] = kv.x; ks[4 * g + 1] = kv.y; ks[4 * g + 2] = kv.z; ks[4 * g + 3] = kv.w;
                        bs[4 * g] = bv.x; bs[4 * g + 1] = bv.y; bs[4 * g + 2] = bv.z; bs[4 * g + 3] = bv.w;
                    }
                    uint32_t (&wv)[4] = wq[h];
                    if (AFFINE) {
                        if (p.relu) requant16_affine<true>(acc[h], ks, bs, wv);
                        else requant16_affine<false>(acc[h], ks, bs, wv);
                    } else {
                        if (p.relu) requant16_fastdiv<true>(acc[h], ks, bs, s_out, inv_s_out, wv);
                        else requant16_fastdiv<false>(acc[h], ks, bs, s_out, inv_s_out, wv);
                    }
                }
                if (valid) {  // 32 channels in one store where the channel count is a multiple of 32
                    if constexpr (NCOLS % 32 == 0) {  // positions are then 32-byte aligned
                        stg32(dst + 32 * hh, wq[0], wq[1]);
                    } else {
#pragma unroll
                        for (int h = 0; h < kPieces; ++h)
                            if (32 * hh + 16 * h < NCOLS)
                                *reinterpret_cast<uint4 *>(dst + 32 * hh + 16 * h) =
                                    make_uint4(wq[h][0], wq[h][1], wq[h][2], wq[h][3]);
                    }
                }
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies in flight land
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == kMmaWarp2) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------

size_t conv_rows_smem_bytes(const ConvRowsParams &q)
{
    const size_t b_bytes = (((size_t)q.taps * q.taps * q.n_cols * q.row_bytes) + 1023) & ~(size_t)1023;
    return 1024 + b_bytes + (size_t)q.n_stages * q.stage_bytes;
}

// Does the kernel serve a conv with `taps` x `taps` stride-1 taps on a grid_h x grid_w grid of
// row_bytes-byte positions and n_total output channels?  Fills what does not depend on the call.
bool conv_rows_plan(int grid_h, int grid_w, int row_bytes, int taps, int n_total, long long max_batch,
                    ConvRowsParams *q)
{
    if ((row_bytes != 32 && row_bytes != 64 && row_bytes != 128) || taps < 1 || taps > 4 || n_total % 16 ||
        n_total < 16 || n_total > 64 || grid_w < taps || grid_h < taps || grid_w > 64)
        return false;
    const int images = 128 / grid_w;
    if (images * grid_w < 108) return false;  // too many idle rows per tile
    if (max_batch * grid_h * grid_w + 512 >= (1LL << 31)) return false;
    memset(q, 0, sizeof(*q));
    q->grid_h = grid_h;
    q->grid_w = grid_w;
    q->row_bytes = row_bytes;
    q->taps = taps;
    q->images = images;
    q->n_cols = n_total;
    // a line's MMAs read 128 rows from each horizontal tap on
    q->stage_bytes = (((128 + taps - 1) * row_bytes) + 1023) & ~1023;
    // stages (input lines): a line takes some 0.3 us, the way from memory under load some 2 us
    for (q->n_stages = kMaxStages2; q->n_stages >= 4; --q->n_stages)
        if (conv_rows_smem_bytes(*q) <= 216 * 1024) return true;
    return false;
}

cudaError_t conv_rows_launch(const void *map_a, const void *map_b, const ConvRowsParams &q0, int batch,
                             int sm_count, cudaStream_t st)
{
    ConvRowsParams q = q0;
    q.batch = batch;
    q.total_lines = (batch + q.images - 1) / q.images * q.out_h;
    const int grid = q.total_lines < sm_count ? q.total_lines : sm_count;
    const size_t smem = conv_rows_smem_bytes(q);
    auto go = [&](auto kernel) -> cudaError_t {
        cudaError_t e = allow_smem((const void *)kernel, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(kThreads2);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, *(const CUtensorMap *)map_a, *(const CUtensorMap *)map_b, q);
    };
    cudaError_t e;
    // (the requantiser is a template parameter, not a branch: both epilogues in one kernel cost time)
    switch (q.n_cols) {
    case 16: e = q.affine ? go(conv_rows_kernel<16, true>) : go(conv_rows_kernel<16, false>); break;
    case 32: e = q.affine ? go(conv_rows_kernel<32, true>) : go(conv_rows_kernel<32, false>); break;
    case 48: e = q.affine ? go(conv_rows_kernel<48, true>) : go(conv_rows_kernel<48, false>); break;
    default: e = q.affine ? go(conv_rows_kernel<64, true>) : go(conv_rows_kernel<64, false>);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace accerl
