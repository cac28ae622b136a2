// Plan of the image-resident residual-network kernels (tc_resnet.cu): does the network have the shape
// they are written for, and if so its weights in their layouts, requantisation constants, buffers, taps.
#include <string.h>

#include <algorithm>

#include "epilogue.cuh"
#include "internal.h"

namespace accerl {

namespace {

// layers 0 .. 17 of the IMPALA network on 84 x 84 frames: per stack conv, pool, two blocks of two convs.  The kernels
// apply ReLU by a layer's number, to what the first conv of a block writes and to what a block reads; that is right
// because networks with other flags are refused here.
bool is_impala(const accerl_layer_desc *layers, int n_layers)
{
    if (n_layers < kResLayers + 2) return false;
    const int channels[3] = {16, 32, 32};
    int c = 4, hw = 84, i = 0;
    auto conv = [&](int n, bool relu_in, bool relu_out, int skip) {
        const accerl_layer_desc &d = layers[i];
        // a ReLU on the input of a layer that reads ReLU'd codes changes nothing
        const bool rin = (d.flags & ACCERL_RELU_IN) && !(i > 0 && (layers[i - 1].flags & ACCERL_RELU_OUT));
        const bool ok = d.kind == ACCERL_CONV2D && d.in_c == c && d.in_h == hw && d.in_w == hw && d.out_c == n && d.kh == 3 &&
                        d.kw == 3 && d.stride == 1 && d.pad == 1 && rin == relu_in &&
                        ((d.flags & ACCERL_RELU_OUT) != 0) == relu_out && d.skip_from == skip;
        c = n;
        ++i;
        return ok;
    };
    for (int s = 0; s < 3; ++s) {
        if (!conv(channels[s], false, false, -1)) return false;
        const accerl_layer_desc &d = layers[i];
        if (d.kind != ACCERL_MAXPOOL || d.kh != 3 || d.kw != 3 || d.stride != 2 || d.pad != 0) return false;
        hw = (hw - 3) / 2 + 1;
        ++i;
        for (int b = 0; b < 2; ++b) {
            const int x = i - 1;
            if (!conv(c, true, true, -1) || !conv(c, false, false, x)) return false;
        }
    }
    for (; i < n_layers; ++i)
        if (layers[i].kind != ACCERL_FC) return false;
    return (layers[kResLayers].flags & ACCERL_RELU_IN) != 0;  // the last block's output is only kept ReLU'd
}

// a layer's requantiser in the kernels' form
void res_layer(const accerl_layer_desc &d, const LayerRequant &rq, ResLayer *L)
{
    memset(L, 0, sizeof(*L));
    for (int c = 0; c < d.out_c; ++c) {
        L->k[c] = rq.k[c];
        L->b[c] = rq.b[c];
        if (d.skip_from >= 0) L->mul[c] = (uint32_t)d.skip_mul[c] << (16 * (c & 1));
    }
    L->s_out = d.s_out;
    L->inv_s_out = rq.inv_s_out;
    L->affine = rq.affine;
}

// byte of K position kk of column n inside a K step's [columns][32 bytes] block, 32-byte swizzle
size_t weight_at(int n, int kk) { return (size_t)n * 32 + (size_t)((((kk >> 4) ^ (n >> 2)) & 1) << 4) + (kk & 15); }

int8_t weight(const accerl_layer_desc &d, int oc, int c, int ky, int kx)
{
    return kx < 0 || kx > 2 ? 0 : d.w[((oc * d.in_c + c) * 3 + ky) * 3 + kx];
}

}  // namespace

accerl_status build_res_steps(accerl_policy *p, const accerl_layer_desc *layers, int n_layers, int8_t **x3,
                              std::vector<Step> *steps, bool *used)
{
    *used = false;
    if (p->in_kind != ACCERL_IN_U8_NCHW || (p->flags & ACCERL_FLAG_TEST_NO_FASTDIV) ||
        !(p->ingest_shift1 || p->ingest_arith == 1) || !is_impala(layers, n_layers))
        return ACCERL_OK;
    ResLayer L[kResLayers];
    for (int i = 0; i < kResLayers; ++i)
        if (layers[i].kind == ACCERL_CONV2D) {
            if (!p->requant[i].fast_div) return ACCERL_OK;
            res_layer(layers[i], p->requant[i], &L[i]);
        }

    // ---- weights
    std::vector<int8_t> w0(kResFirstWeights, 0), w1(kRes1Weights, 0), w2(kRes2Weights, 0);
    for (int ky = 0; ky < 3; ++ky)  // columns: five output pixels 4X - 2 ..; K: pixels 4X - 4 .. 4X + 3
        for (int px = 0; px < 5; ++px)
            for (int oc = 0; oc < 16; ++oc)
                for (int kk = 0; kk < 32; ++kk)
                    w0[(size_t)ky * 80 * 32 + weight_at(px * 16 + oc, kk)] = weight(layers[0], oc, kk % 4, ky, kk / 4 - px - 1);
    for (int op = 0; op < 6; ++op)  // columns: two output pixels; K steps: pixel pairs (0, 1) and (2, 3) of each line
        for (int j = 0; j < 6; ++j)
            for (int px = 0; px < 2; ++px)
                for (int oc = 0; oc < 16; ++oc)
                    for (int kk = 0; kk < 32; ++kk)
                        w1[(size_t)(op * 6 + j) * 1024 + weight_at(px * 16 + oc, kk)] =
                            weight(layers[op < 4 ? 2 + op : 6], op == 5 ? 16 + oc : oc, kk % 16, j / 2, 2 * (j % 2) + kk / 16 - px);
    const int of_op[9] = {8, 9, 10, 11, 12, 14, 15, 16, 17};
    for (int op = 0; op < 9; ++op)
        for (int j = 0; j < 9; ++j)
            for (int oc = 0; oc < 32; ++oc)
                for (int kk = 0; kk < 32; ++kk)
                    w2[(size_t)(op * 9 + j) * 1024 + weight_at(oc, kk)] = weight(layers[of_op[op]], oc, kk, j / 3, j % 3);
    void *d0 = nullptr, *d1 = nullptr, *d2 = nullptr;
    accerl_status st = upload_bytes(p, w0.data(), w0.size(), &d0);
    if (st == ACCERL_OK) st = upload_bytes(p, w1.data(), w1.size(), &d1);
    if (st == ACCERL_OK) st = upload_bytes(p, w2.data(), w2.size(), &d2);
    if (st != ACCERL_OK) return st;

    // ---- the tensors between the kernels
    const size_t mb = (size_t)p->max_batch, bytes[3] = {mb * kRes1Bytes, mb * kRes2Bytes, mb * kRes3Bytes};
    int8_t *x[3];
    for (int i = 0; i < 3; ++i) {
        void *d = nullptr;
        ACCERL_CUDA_TRY(device_alloc(&d, bytes[i] + 4096));
        p->owned.push_back(d);
        p->workspace_bytes += bytes[i] + 4096;
        x[i] = (int8_t *)d;
    }
    *x3 = x[2];

    ResFirstParams &f = p->res_first;
    f.w = (const uint8_t *)d0;
    f.x1 = x[0];
    f.ingest_mode = p->ingest_shift1 ? 2 : 1;
    f.ingest_mul = p->ingest_mul;
    f.ingest_add = p->ingest_add;
    f.status = p->status_word;
    f.layer = L[0];
    ResStack1Params &a = p->res_stack1;
    a.x1 = x[0];
    a.w = (const uint8_t *)d1;
    a.x2 = x[1];
    a.status = p->status_word;
    for (int i = 0; i < 5; ++i) a.layer[i] = L[2 + i];
    ResStack23Params &b = p->res_stack23;
    b.x2 = x[1];
    b.w = (const uint8_t *)d2;
    b.x3 = x[2];
    b.status = p->status_word;
    for (int i = 0; i < 9; ++i) b.layer[i] = L[of_op[i]];
    if (p->flags & ACCERL_FLAG_KEEP_ACTIVATIONS) {  // (with TAP_FUSED) plain copies of what the kernels compute
        auto buf = [&](int layer) { return p->bufs[p->layers[layer].out_buf].ptr; };
        f.tap_in = p->bufs[p->layers[0].in_buf].ptr;
        f.tap_x1 = buf(1);
        for (int i = 0; i < 4; ++i) a.tap[i] = buf(2 + i);
        a.tap_x2 = buf(7);
        for (int i = 0; i < 8; ++i) b.tap[i] = buf(of_op[i]);
        b.tap_x3 = buf(13);
        for (int t : {0, 6, 17}) p->tap_missing[t + 1] = 1;  // pooled before, or kept ReLU'd only
    }

    auto note = [&](int lo, int hi) {
        bool affine = false, division = false;
        for (int i = lo; i <= hi; ++i)
            if (layers[i].kind == ACCERL_CONV2D) (L[i].affine ? affine : division) = true;
        return std::string(affine ? "[single-fma requantiser verified]" : "") + (division ? "[3-step divide verified]" : "");
    };
    auto add = [&](Step::Kind kind, const std::string &kernel, const char *covers) {
        Step s;
        s.kind = kind;
        s.kernel = kernel;
        s.covers = covers;
        steps->push_back(s);
    };
    add(Step::RES_FIRST, "res_first_kernel" + note(0, 0) + "[frames quantised inside][pooled along x on the accumulators]",
        "ingest+layers 0-1");
    add(Step::RES_STACK1, "res_stack1_kernel" + note(2, 6), "layers 2-7");
    add(Step::RES_STACK23, "res_stack23_kernel" + note(8, 17), "layers 8-17");
    *used = true;
    return ACCERL_OK;
}

}  // namespace accerl
