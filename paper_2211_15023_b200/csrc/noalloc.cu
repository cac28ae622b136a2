// accerl_policy_act_noalloc: the Actor step for callers that must not allocate device memory.
//
// The activation workspace of this variant is a fixed array inside the library image instead of
// buffers obtained from cudaMalloc.  See the declaration in accerl.h for who needs it and why.
#include <algorithm>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace {

constexpr size_t kScratchBytes = ACCERL_NOALLOC_SCRATCH_BYTES;
constexpr int kMaxDevices = 64;

// Reserved on every GPU on which this library's CUDA module gets loaded, until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_mu;
unsigned char *g_scratch_dev[kMaxDevices];  // device address of the array, per device; null = not yet asked

struct CurrentDevice {
    int prev = -1;
    bool ok;
    explicit CurrentDevice(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        ok = prev == dev || cudaSetDevice(dev) == cudaSuccess;
        if (prev == dev) prev = -1;
    }
    ~CurrentDevice()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// In host code `g_noalloc_scratch` is only a handle for the runtime, not an address a kernel can
// use: ask the runtime once per device (with that device current) where the array lives there.
accerl_status scratch_on(int device, unsigned char **out)
{
    if (device < 0 || device >= kMaxDevices) {
        accerl::set_error("act_noalloc: device index %d not supported (0..%d)", device,
                          kMaxDevices - 1);
        return ACCERL_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_dev[device]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess || !ptr) {
            accerl::set_error("act_noalloc: cudaGetSymbolAddress failed on device %d: %s", device,
                              cudaGetErrorString(e));
            cudaGetLastError();
            return ACCERL_ERR_CUDA;
        }
        g_scratch_dev[device] = (unsigned char *)ptr;
    }
    *out = g_scratch_dev[device];
    return ACCERL_OK;
}

using namespace accerl;

// The policy's own plan on the fixed array: a copy of the handle whose activation pointers and TMA maps
// lead there.  Weights, scales and the status word are the handle's; nothing is allocated on the device.
// (Stepping through the CUDA-core kernels instead took 182 us for 160 states of the Nature-CNN.)
// Null when the plan keeps tensors whose borders must stay zero, or taps.
std::unique_ptr<accerl_policy> make_twin(accerl_policy *p, unsigned char *base)
{
    if (p->flags & (ACCERL_FLAG_KEEP_ACTIVATIONS | ACCERL_FLAG_FORCE_GENERIC)) return nullptr;
    bool resident = false;
    for (const Step &s : p->steps) {
        switch (s.kind) {
        case Step::RES_FIRST: resident = true; break;
        case Step::RES_STACK1: case Step::RES_STACK23: case Step::MLP_FUSED: case Step::CONV1_FRAMES: case Step::CONV_ROWS: case Step::ATARI:
        case Step::FC_SAMPLE: case Step::FC_HEAD: case Step::FC_TILE: case Step::SAMPLE: break;
        case Step::TC_GEMM: {
            const TcGemmParams &g = p->tc_steps[s.tc].prm;  // no padded layouts, no residual or second output
            if (g.out2 || g.skip || g.px_per_row || g.out_row_off) return nullptr;
            break;
        }
        default: return nullptr;
        }
    }
    // activation regions of the plan, as bytes per state
    struct Region {
        const char *old_base;
        size_t per_state;
        char *new_base;
    };
    std::vector<Region> regions;
    if (!p->mlp)
        for (size_t b = 0; b < p->bufs.size(); ++b) {
            // (the resident kernels leave the conv layers' buffers unused)
            bool used = !resident;
            for (size_t i = kResLayers; i < p->layers.size() && !used; ++i) used = p->layers[i].out_buf == (int)b;
            if (used) regions.push_back(Region{(const char *)p->bufs[b].ptr, p->bufs[b].bytes_per_state, nullptr});
        }
    if (p->z_scratch) regions.push_back(Region{(const char *)p->z_scratch, (size_t)p->n_out * sizeof(float), nullptr});
    if (resident) {
        regions.push_back(Region{(const char *)p->res_first.x1, kRes1Bytes, nullptr});
        regions.push_back(Region{(const char *)p->res_stack1.x2, kRes2Bytes, nullptr});
        regions.push_back(Region{(const char *)p->res_stack23.x3, kRes3Bytes, nullptr});
    }
    size_t per_state = 0;
    for (const Region &r : regions) per_state += r.per_state;
    // the largest batch the regions fit, each rounded up to 1 KB (TMA boxes may start in the last rows)
    size_t cap = (size_t)INT32_MAX;  // the single-launch MLP keeps no activations
    if (per_state) cap = std::min<size_t>(4096, (kScratchBytes - 1024 * regions.size()) / per_state);
    size_t at = 0;
    for (Region &r : regions) {
        r.new_base = (char *)base + at;
        at += (r.per_state * cap + 1023) / 1024 * 1024;
    }
    std::unique_ptr<accerl_policy> q(new accerl_policy(*p));
    q->noalloc_twin = nullptr;
    q->owned.clear();
    q->events.clear();
    q->copy_events.clear();
    q->copy_stream = nullptr;
    q->mix = SideStream();
    q->ptq.clear();
    q->ptq_data.reset();
    q->max_batch = (int)cap;
    bool ok = true;
    auto move = [&](auto *&ptr) {
        if (!ptr) return;
        for (const Region &r : regions)
            if ((const char *)ptr >= r.old_base && (const char *)ptr < r.old_base + r.per_state * (size_t)p->max_batch + 256) {
                ptr = (std::remove_reference_t<decltype(ptr)>)(r.new_base + ((const char *)ptr - r.old_base));
                return;
            }
        ok = false;
    };
    auto remap = [&](void *map, ActivationMap &m) {
        move(m.base);
        if (ok && tc_make_map(map, m.base, m.rows_per_state * (long long)cap, m.row_bytes, m.pitch, m.box_rows, m.box_bytes) != ACCERL_OK)
            ok = false;
    };
    for (const Step &s : q->steps) {
        if (s.kind == Step::TC_GEMM) {
            TcStep &t = q->tc_steps[s.tc];
            if (!t.prm.fuse_ingest) remap(t.map_a, t.a_map);  // (that one reads the frames themselves)
            if (!t.prm.logits_mode) move(t.prm.out);
        } else if (s.kind == Step::CONV_ROWS) {
            ConvRowsStep &c = q->conv_rows[s.tc];
            remap(c.map_a, c.a_map);
            move(c.prm.out);
        } else if (s.kind == Step::CONV1_FRAMES) {
            move(q->conv1.out);
        } else if (s.kind == Step::ATARI) {
            move(q->atari.out);
        } else if (s.kind == Step::FC_HEAD) {
            move(q->fc_head.x);
        } else if (s.kind == Step::FC_TILE) {
            remap(q->fc_tile_map, q->fc_tile_a);
        } else if (s.kind == Step::FC_SAMPLE) {
            move(q->fc_sample.x);
        } else if (s.kind == Step::RES_FIRST) {
            move(q->res_first.x1);
            move(q->res_stack1.x1);
            move(q->res_stack1.x2);
            move(q->res_stack23.x2);
            move(q->res_stack23.x3);
        }
    }
    move(q->z_scratch);
    if (!ok) q.reset();
    return q;
}

// made once per handle; null for good where there is none, or no host memory for it
accerl_policy *twin_of(accerl_policy *p, unsigned char *base)
{
    std::lock_guard<std::mutex> lock(g_mu);
    if (!p->noalloc_tried) {
        p->noalloc_tried = true;
        try {
            p->noalloc_twin = make_twin(p, base).release();
        } catch (const std::bad_alloc &) {
        }
    }
    return p->noalloc_twin;
}

}  // namespace

extern "C" accerl_status accerl_policy_act_noalloc(accerl_policy *p, const void *obs_dev,
                                                   const float *uniforms_dev, int32_t batch,
                                                   float *logits_dev, int32_t *actions_dev,
                                                   float *logp_dev, void *cuda_stream)
{
    if (!p || !obs_dev || !uniforms_dev || !logits_dev || !actions_dev || !logp_dev) {
        set_error("act_noalloc: null argument");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (batch < 1) {
        set_error("act_noalloc: batch must be at least 1");
        return ACCERL_ERR_INVALID_ARG;
    }
    if (((uintptr_t)obs_dev & 15) || ((uintptr_t)uniforms_dev & 3) || ((uintptr_t)logits_dev & 3) ||
        ((uintptr_t)actions_dev & 3) || ((uintptr_t)logp_dev & 3)) {
        set_error("act_noalloc: misaligned pointer (obs needs 16 bytes, the others 4)");
        return ACCERL_ERR_INVALID_ARG;
    }
    // carve the handle's logical buffers out of the fixed array
    constexpr int kMaxBufs = 64;
    size_t offset[kMaxBufs];
    if (p->bufs.size() > (size_t)kMaxBufs) {
        set_error("act_noalloc: the policy needs %zu workspace buffers (at most %d supported)",
                  p->bufs.size(), kMaxBufs);
        return ACCERL_ERR_UNSUPPORTED;
    }
    size_t total = 0;
    for (size_t b = 0; b < p->bufs.size(); ++b) {
        offset[b] = total;
        size_t bytes = p->bufs[b].bytes_per_state * (size_t)batch;
        total += (bytes + 255) / 256 * 256;
    }
    // a value head: the last layer's rows (logits, then V) pass through the array as well
    const size_t z_offset = total;
    if (p->n_out != p->n_actions) total += ((size_t)batch * p->n_out * sizeof(float) + 255) / 256 * 256;
    if (total > kScratchBytes) {
        set_error("act_noalloc: batch %d needs %zu bytes of activation workspace, the built-in "
                  "scratch holds %zu (use accerl_policy_act, or a smaller batch)",
                  batch, total, kScratchBytes);
        return ACCERL_ERR_BATCH_TOO_LARGE;
    }
    CurrentDevice cur(p->device);
    if (!cur.ok) {
        set_error("act_noalloc: cudaSetDevice(%d) failed", p->device);
        return ACCERL_ERR_CUDA;
    }
    unsigned char *base = nullptr;
    accerl_status s = scratch_on(p->device, &base);
    if (s != ACCERL_OK) return s;
    if (accerl_policy *twin = twin_of(p, base); twin && batch <= twin->max_batch) {
        p->last_stream = (cudaStream_t)cuda_stream;  // accerl_policy_check waits for this step
        return run_steps(twin, obs_dev, uniforms_dev, batch, logits_dev, actions_dev, logp_dev, nullptr, nullptr,
                         (cudaStream_t)cuda_stream, nullptr);
    }
    // a plan that cannot be moved, or a batch beyond its share of the array: the CUDA-core kernels
    auto buf = [&](int b) { return (int8_t *)(base + offset[b]); };

    cudaStream_t st = (cudaStream_t)cuda_stream;
    p->last_stream = st;  // accerl_policy_check waits for this step
    const int B = batch;
    float *z_dev = p->n_out != p->n_actions ? (float *)(base + z_offset) : logits_dev;
    int8_t *x = buf(p->layers[0].in_buf);
    if (p->in_kind == ACCERL_IN_U8_NCHW)
        ACCERL_CUDA_TRY(launch_ingest_u8((const uint8_t *)obs_dev, p->lut, x, B, p->in_c, p->in_h,
                                         p->in_w, p->in_cp, st));
    else
        ACCERL_CUDA_TRY(launch_ingest_f32((const float *)obs_dev, p->s_input, x, B, p->in_c,
                                          p->in_cp, st));
    for (const LayerPlan &L : p->layers) {
        const int8_t *in = buf(L.in_buf);
        int8_t *o = L.out_buf >= 0 ? buf(L.out_buf) : nullptr;
        if (L.kind == ACCERL_CONV2D)
            ACCERL_CUDA_TRY(launch_conv_generic(L, in, L.skip_buf >= 0 ? buf(L.skip_buf) : nullptr, o,
                                                B, st));
        else if (L.kind == ACCERL_FC)
            ACCERL_CUDA_TRY(launch_fc_generic(L, in, o, z_dev, B, st));
        else
            ACCERL_CUDA_TRY(launch_maxpool_generic(L, in, o, B, st));
    }
    ACCERL_CUDA_TRY(launch_sample(z_dev, p->n_out, uniforms_dev, B, p->n_actions,
                                  z_dev != logits_dev ? logits_dev : nullptr, actions_dev, logp_dev,
                                  nullptr, nullptr, st));
    return ACCERL_OK;
}
