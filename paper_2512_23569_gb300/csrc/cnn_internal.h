// The learned noise-level network's handle and the entry points shared by its
// two translation units: cnn.cu (FP32 forward and backward for training,
// Adam, readout, host interface) and cnn_tc.cu (the tensor-core forward pass
// used for denoising).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "hts_internal.h"

struct hts_cnn {
    int C = 1, device = 0, nparams = 0, t = 0, window = 128;
    int off[5] = {}, cin[5] = {}, cout[5] = {};  // per layer: parameter offset, input / output channels
    float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;  // FP32 parameters, Adam state
    __half *w16 = nullptr;                                                  // FP16 copy used by the kernels
    // the tensor-core kernels' weights, FP16, laid out as their shared memory holds them ([tap][plane][n][8], zero
    // outside the layer's channels): layer l's at wpk + pf[l], and for l >= 1 the flipped, transposed ones of the
    // backward pass at wpk + pb[l]; written with w16
    __half *wpk = nullptr;
    int pf[5] = {}, pb[5] = {}, npk = 0;
    size_t cap_px = 0;
    float *act[5] = {};                   // FP32 activations (planar CHW) of the training forward
    float *d0 = nullptr, *d1 = nullptr;   // gradient maps; d0 also holds the readout's row sums
    size_t cap_part = 0;
    float *part = nullptr;                // per-tile partial weight gradients
    double *loss = nullptr;
    size_t cap_h16 = 0, cap_map = 0, cap_rows = 0;
    __half *h16[2] = {};    // FP16 activations of the tensor-core forward, 4 planes of 8 channels
    float *map = nullptr;   // its log-sigma map (H x W)
    float *rows = nullptr;  // row sums of the readout window (H x reference columns)
    int *err = nullptr;     // set by a tensor-core forward whose wait gave up (the map is then NaN)
    double *lpart = nullptr;  // the loss kernel's per-block parts (LOSS_BLOCKS), then its block counter
    // tensor-core training (cnn_tc.cu): per-layer FP16 activations, the FP16 gradients of the hidden layers'
    // outputs, the map and its loss gradient, per-block weight-gradient sums
    int train_tc = 1;  // 1: hts_cnn_accumulate_grad runs on the tensor cores (FP16); 0: the FP32 kernels
    size_t tr_cap_px = 0, tr_cap_part = 0;
    __half *tr_act[4] = {}, *tr_dy[4] = {};
    float *tr_map = nullptr, *tr_d0 = nullptr, *tr_part = nullptr;
};

namespace hts {

// Tensor-core forward pass (cnn_tc.cu): the log-sigma map of img (device,
// planar C x H x W, [0, 255]) in map (H x W, FP32).  Hidden activations are
// rounded to FP16 (8-channel planes, in h0 and h1: H * W * 32 halves each), the
// network input x / 255 too; FP16 weights, FP32 accumulation in tensor memory.
// Only the weights and the error flag are the net's.
hts_status cnn_forward_tc_into(hts_cnn *net, const float *img, int H, int W, __half *h0, __half *h1, float *map,
                               cudaStream_t s);
// The net's own buffers: its activations h16; those, its map and its rows (for nx reference columns).
hts_status cnn_ensure_h16(hts_cnn *net, int H, int W);
hts_status cnn_ensure_infer(hts_cnn *net, int H, int W, int nx);
struct Geom;
// Training loss (added to net->loss) of the map over the reference patches and its gradient map (dout, every pixel).
hts_status cnn_loss(hts_cnn *net, const float *map, int H, int W, const Geom &g, const float *target, float *dout,
                    cudaStream_t s);
constexpr int LOSS_BLOCKS = 304;
// One image's loss and gradient (added to net->grad) on the tensor cores: FP16 activations and input
// gradients (loss scale 2^(floor(log2 N_ref) + 2)), FP32 accumulation of the weight gradients.
hts_status cnn_grad_tc(hts_cnn *net, const float *img, int H, int W, const Geom &g, const float *target,
                       cudaStream_t s);
// Noise level of every reference patch (sigma_ref, device, N_ref) through the
// readout window, from a forward into caller-owned buffers (rows: H * nx floats).
hts_status cnn_sigma_refs_into(hts_cnn *net, const float *img, const Geom &g, __half *h0, __half *h1, float *map,
                               float *rows, float *sigma_ref, cudaStream_t s);

}  // namespace hts
