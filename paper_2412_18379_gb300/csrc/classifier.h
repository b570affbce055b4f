// The classifier start predictor (Sec. 2.3, Eq. 7-8): shapes and the
// launchers of its non-GEMM kernels (internal).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "fc_tc.h"
#include "internal.h"

namespace cs {

constexpr int kClsCh = 32;     // channels of both convolutions
constexpr int kClsH1 = 256;    // width of the offset branch (h1, Sec. 3.1)
constexpr int kClsH2 = 512;    // width of the fused layer (h2, Sec. 3.1)

inline int cls_window(int dim) { return dim == 2 ? 9 : 7; }
inline int cls_cells(int dim) {           // W^dim: window cells = classes
    const int W = cls_window(dim);
    return dim == 2 ? W * W : W * W * W;
}
inline int cls_pooled(int dim) {          // 32 (W/2)^dim pooled features
    const int p = cls_window(dim) / 2;
    return kClsCh * (dim == 2 ? p * p : p * p * p);
}

void launch_departure(int64_t n, int dim, const double *x, const double *u, double dt,
                      double *xp, int sm_count, cudaStream_t st);
// window [B][dim][E^dim] (E = W, or W + 2 with a zero ring when pad) and
// offset [B][dim] of the particles xp[idx[b]] (idx may be null: b)
void launch_cls_features(const DevMesh &m, int64_t B, const double *xp, const int64_t *idx,
                         bool pad, float *win, float *offset, int sm_count, cudaStream_t st);
void launch_cls_pad(int dim, const float *y, int64_t B, int C, float *a, int sm_count,
                    cudaStream_t st);
void launch_cls_crop_relu_back(int dim, const float *dpad, const float *z, int64_t B, int C,
                               float *dz, int sm_count, cudaStream_t st);
void launch_cls_pool(int dim, const float *z, int64_t B, float *cat, int64_t ldc, int sm_count,
                     cudaStream_t st);
void launch_cls_pool_back(int dim, const float *dcat, int64_t ldc, const float *z, int64_t B,
                          float *dz, int sm_count, cudaStream_t st);
void launch_cls_cat_relu(const float *y, int64_t B, int n, float *cat, int64_t ldc, int64_t off,
                         int sm_count, cudaStream_t st);
void launch_cls_uncat_relu_back(const float *dcat, int64_t ldc, int64_t off, const float *y,
                                int64_t B, int n, float *dy, int sm_count, cudaStream_t st);
void launch_softmax_ce(const float *H, const int32_t *labels, const int64_t *idx, int64_t B,
                       int n_cls, float *dH, float *loss, cudaStream_t st);
void launch_cls_labels(const DevMesh &m, int64_t n, const double *xp, const int32_t *host,
                       int32_t *label, int sm_count, cudaStream_t st);
// start[i] (user ids) and class of rows i < n from their logits; fallback
// null means the plain start of mesh node row0 + i
void launch_cls_start(const DevMesh &m, int64_t n, const double *xp, const float *logits,
                      const int32_t *fallback, int64_t row0, int32_t *start, int32_t *cls,
                      int sm_count, cudaStream_t st);

// module 1 fused on the tensor cores (classifier_tc.cu): conv1 and conv2
// weights packed for the kernel (bytes, and the packing from the FP32
// parameters), then per particle the window inputs, both convolutions and the
// pooling into the first 32 (W/2)^dim columns of cat (BF16 tiled, fc_tc.h) and
// the offset into off[b][dim]. pool_f: the mesh's pooled centroids as float hi + lo.
int64_t cls_packed_bytes(int dim);
void launch_cls_pack(int dim, const float *w, int64_t off_w1, int64_t off_b1, int64_t off_w2,
                     int64_t off_b2, uint8_t *packed, cudaStream_t st);
void launch_cls_conv_tc(const DevMesh &m, const float *pool_f, int64_t B, const double *xp,
                        const uint8_t *packed, const FcMat &cat, float *off, int *err,
                        int sm_count, cudaStream_t st);

// Training on the tiled layouts (classifier.cu).
// The pooled ReLU(z) of pool_relu as BF16 into cat's first columns (zero rows past B)
void launch_cls_pool_tiled(int dim, const float *z, int64_t B, const FcMat &cat, int sm_count,
                           cudaStream_t st);
// the pooling's gradient through the second ReLU: dz[b][p][c] BF16 from
// dpool [B][32 (W/2)^dim], and its column sums part[block][32], blocks =
// cls_pool_back_blocks
int cls_pool_back_blocks(int64_t B, int sm_count);
void launch_cls_pool_back_tiled(const float *dpool, const float *z, int64_t B, uint16_t *dz,
                                float *part, int sm_count, cudaStream_t st);
// softmax and cross-entropy gradient (softmax_ce) into the tiled gH (n_cls
// columns rounded up to 16, zero padding), column sums and loss sums per block:
// part[block][n_cls], loss_part[block], blocks = cls_softmax_blocks(B); the
// loss is the sum over n_valid, a count left in *count
int cls_softmax_blocks(int64_t B);
void launch_softmax_ce_tiled(const float *H, const int32_t *labels, const int64_t *idx, int64_t B,
                             int n_cls, const FcMat &gH, float *part, float *loss_part, int *count,
                             cudaStream_t st);
// *loss = sum of n loss_part / *count (0 where that is 0)
void launch_loss_sum(const float *loss_part, int n, const int *count, float *loss, cudaStream_t st);

}  // namespace cs
