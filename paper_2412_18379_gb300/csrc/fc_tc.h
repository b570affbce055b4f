// Fully connected layers on BF16 operands in tiled layouts (fc_tc.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

namespace cs {

// A tiled BF16 matrix of M rows and K columns (K a multiple of 16): row tiles
// of 128, each [K / 8][128][8], the operand layout of the MMA, so a K range of
// a row tile is one contiguous block. Rows past M up to the tile's end exist.
struct FcMat {
    uint8_t *p = nullptr;
    int64_t tile = 0;             // bytes per row tile
    int chunk0 = 0;               // first 8-column chunk of the matrix in the tile
    int chunks = 0;               // K / 8
};
constexpr int64_t kFcChunk = 128 * 16;
inline int64_t fc_bytes(int64_t M, int K) { return (M + 127) / 128 * (K / 8) * kFcChunk; }
inline FcMat fc_mat(uint8_t *p, int K) { return FcMat{p, (K / 8) * kFcChunk, 0, K / 8}; }
// columns [c0, c0 + n) of a matrix (multiples of 8)
inline FcMat fc_cols(FcMat m, int c0, int n) {
    m.chunk0 += c0 / 8;
    m.chunks = n / 8;
    return m;
}

// A weight matrix R(r, k) = W[r rs + k ks], r < rows, k < K, as the right operand
// of fc_gemm: BF16 [row tiles of BN][Kp / 8][BN][8], zero past the rows and past K
struct FcPack {
    const float *W;
    int64_t rs, ks;
    int rows, K, BN;
    uint8_t *out;
};
constexpr int kMaxFcPack = 12;
inline int fc_kp(int K) { return (K + 15) / 16 * 16; }
inline int64_t fc_packed_bytes(int rows, int K, int BN) {
    return int64_t((rows + BN - 1) / BN) * BN * fc_kp(K) * 2;
}
// columns per CTA tile of a product of M rows and N columns: wide tiles read
// their operands least often, but few rows then leave SMs idle
int fc_bn(int64_t M, int N, int sm_count);
int launch_fc_pack(const FcPack *segs, int n, cudaStream_t st);

// v(i, j) = sum_k A(i, k) R(j, k) (+ bias[j]), j < N, i < M, in K order with
// K = 16 steps (the general GEMM's bits for an unsplit K). Then, as given:
// relu; gate: v = gate(i, j) > 0 ? v : 0; out: BF16 tiled (zero rows past M);
// f32: row-major [M][ldf]; colsum: partial column sums [4 ceil(M / 128)][N] of v.
struct FcGemm {
    FcMat A;
    const uint8_t *B;
    int BN, N;
    int64_t M;
    const float *bias = nullptr;
    bool relu = false;
    FcMat gate;
    FcMat out;
    float *f32 = nullptr;
    int64_t ldf = 0;
    float *colsum = nullptr;
    // K splits: partial sums of kc columns each (a multiple of 64), added in
    // order; BN <= 128 then
    int nsplit = 1, kc = 0;
};
// the general GEMM's split of a product with bias (tc_gemm.cu), whose bits an
// emulating product must give: splits, and columns per split
void fc_split_like_gemm(int64_t M, int N, int K, int sm_count, int *nsplit, int *kc);
int launch_fc_gemm(const FcGemm &g, int *err, int sm_count, cudaStream_t st);

// part[s][n][k] = sum over the rows of split s of Y(row, n) X(row, k), n < N, k < K:
// weight gradients; both operands' rows past M are zero
int fc_wgrad_splits(int64_t M, int N, int K, int sm_count);
int launch_fc_wgrad(const FcMat &Y, const FcMat &X, int64_t M, int N, int K, int splits,
                    float *part, int *err, cudaStream_t st);

// out[i][c] = FP32 of A(i, c), row-major with row stride ld, i < M
int launch_fc_widen(const FcMat &A, int64_t M, float *out, int64_t ld, cudaStream_t st);

// r[i][n] = BF16 of ReLU(sum_d BF16(off[i][d]) BF16(W[n][d]) + b[n]), n < 256, tiled
int launch_fc_offset(int dim, int64_t M, const float *off, const float *W, const float *b,
                     const FcMat &r, int sm_count, cudaStream_t st);
// part[t][256 dim]: over row tile t, the weight gradient of that layer from gy
int launch_fc_offset_grad(int dim, int64_t M, const float *off, const FcMat &gy, float *part,
                          cudaStream_t st);

}  // namespace cs
