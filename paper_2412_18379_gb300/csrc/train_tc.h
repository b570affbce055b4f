// Fused training kernels of the convolutional networks (train_tc.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace cs {

constexpr int kTrainCh = 32;      // channels of every convolution

// One valid 3^D convolution of 32 output channels over B inputs of edge Si.
struct ConvGeo {
    int dim, C, Si;               // C input channels
    int So, Pi, Po, K;            // output edge, positions, K = C 3^D
    ConvGeo(int d, int c, int si) : dim(d), C(c), Si(si) {
        So = si - 2;
        Pi = d == 2 ? si * si : si * si * si;
        Po = d == 2 ? So * So : So * So * So;
        K = c * (d == 2 ? 9 : 27);
    }
};

// Packed weights of a training step: per convolution W[32][K] -> fwd (BF16
// [Kp / 8][32][8], Kp = K rounded up to 16) and bwd (BF16 [4][kw][8], row 32 tap +
// channel); fc1's W1[256][32] -> fc1 (BF16 [4][256][8]). Null outputs are skipped.
struct PackSeg {
    const float *W;
    int K, kw;
    uint8_t *fwd, *bwd, *fc1;
};
constexpr int kMaxPack = 6;
int train_packed_kw(int dim);     // rows of bwd
int launch_pack_train(const PackSeg *segs, int n, cudaStream_t st);

// y = BF16 of ReLU(conv(x) + bias). x: BF16 [B][Pi][32], or FP32 channels
// first [B][C][Pi] when `first`. y (may be null): BF16 [B][edge^D][32] with
// the output position (px, ..) at (px + ring, ..), edge = So + 2 ring; z (may
// be null): FP32 conv(x) + bias [B][Po][32]. packed: PackSeg::fwd.
int launch_conv_fwd(const ConvGeo &g, const void *x, bool first, int64_t B, const uint8_t *packed,
                    const float *bias, uint16_t *y, int ring, float *z, int *err, int sm_count,
                    cudaStream_t st);

// CTAs of launch_conv_bwd (one partial of every gradient each)
int conv_bwd_ctas(const ConvGeo &g, int64_t B, bool first, int sm_count);
// Weight gradient partials of one convolution, wpart[cta][32 K] (the weights'
// layout), from its input x (as in launch_conv_fwd) and its output gradient dz
// (BF16 [B][Po][32]); and, except for the first layer, its input's gradient
// through the ReLU (x > 0): dzp BF16 [B][Pi][32] (Si = 11: x has a zero ring that
// dzp leaves out, [B][81][32]), and the column sums of its FP32 values
// bpart[cta][32]. packed: PackSeg::bwd.
int launch_conv_bwd(const ConvGeo &g, const void *x, bool first, int64_t B, const uint16_t *dz,
                    const uint8_t *packed, float *wpart, uint16_t *dzp, float *bpart, int *err,
                    int sm_count, cudaStream_t st);

// The regressor's head on h [B][32] (BF16): out = W2 ReLU(W1 h + b1) + b2 (FP32
// [B][dim]). With targets also the mean squared error's gradients: dz [B][32]
// (BF16, through h > 0), and partials per CTA: W1 [256 32], b1 [256], W2
// [dim 256], b2 [dim], the bias sums of dz [32] and the squared error [1],
// head_part_floats(dim) floats in that order.
int head_ctas(int64_t B, int sm_count);
int64_t head_part_floats(int dim);
int launch_train_head(int dim, int64_t B, const uint16_t *h, const uint8_t *packed_w1,
                      const float *b1, const float *W2, const float *b2, const float *tgt,
                      float *out, uint16_t *dz, float *part, int *err, int sm_count,
                      cudaStream_t st);

// out[i] = sum over p < n, in a fixed order, of part[p stride + i] for i < count,
// divided by `div` where that is > 0
struct ReduceSeg {
    const float *part;
    int64_t stride, count;
    float *out;
    int n;
    float div;
};
constexpr int kMaxSegs = 16;
int launch_reduce_parts(const ReduceSeg *segs, int n_segs, cudaStream_t st);

}  // namespace cs
