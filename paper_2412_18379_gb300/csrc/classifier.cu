// The paper's classifier start predictor (Sec. 2.3, Eq. 7-8): the kernels
// around its layers' products. Inputs (pooled centroid windows and the offset of
// x_p), average pooling and its gradient, the softmax with its cross-entropy
// gradient, each on the tiled BF16 layouts (fc_tc.h) and, for FP32 operands and
// batches below 16 rows, on row-major FP32 with the zero padding and concatenation
// that path needs; the labels from plain SNS hosts and the start element K_p of
// the most probable class.
//
// Every FP64 step of the inputs, labels and starts is written with explicit
// round-to-nearest intrinsics, so the integer decisions (cells, labels,
// starts) and the FP64 feature values are those of a plain evaluation of the
// same formulas; the network itself runs in BF16/FP32 (classifier.cpp).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "classifier.h"
#include "walk_common.cuh"

namespace cs {
namespace {

constexpr int kT = 256;

int blocks_for(int64_t n, int sm_count, int per_sm = 16) {
    const int64_t b = (n + kT - 1) / kT;
    return int(std::max<int64_t>(1, std::min<int64_t>(b, int64_t(sm_count) * per_sm)));
}

template <int D>
struct Win {
    static constexpr int W = D == 2 ? 9 : 7;        // window edge
    static constexpr int P = D == 2 ? W * W : W * W * W;
    static constexpr int Wq = W + 2;                 // zero-padded edge
    static constexpr int Pq = D == 2 ? Wq * Wq : Wq * Wq * Wq;
    static constexpr int Wp = W / 2;                 // pooled edge (odd row dropped)
    static constexpr int Pp = D == 2 ? Wp * Wp : Wp * Wp * Wp;
};

// x_p = x - (u * dt) (Eq. 3)
__global__ void departure_kernel(int64_t n, const double *__restrict__ x,
                                 const double *__restrict__ u, double dt,
                                 double *__restrict__ xp) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x)
        xp[i] = __dsub_rn(x[i], __dmul_rn(u[i], dt));
}

// float(a / s) with the quotient rounded to FP64 first, without the FP64
// division (some 25 instructions of the pipe that every FP64 instruction
// holds for ~56 cycles per warp): a * (1 / s) is within 2 ulp of it, so both
// round to the same float unless a rounding boundary (the midpoint of two
// floats: the 29 dropped bits at 2^28) lies that close; those values, and
// those outside the normal floats, take the division.
__device__ __forceinline__ float quotient_to_float(double a, double s, double inv) {
    const double q = __dmul_rn(a, inv);
    uint32_t lo, hi;
    dbits(q, lo, hi);
    const int E = int((hi >> 20) & 0x7ffu) - 1023;
    const int tail = int(lo & 0x1fffffffu) - 0x10000000;
    if (((hi << 1) | lo) == 0 || (E >= -126 && E < 127 && (tail > 16 || tail < -16)))
        return __double2float_rn(q);
    return __double2float_rn(__ddiv_rn(a, s));
}

// Cell of one axis: the FP64 formula's, certified in FP32 (grid_cell_cert's
// test) where the rounding bound cannot move the quotient across an integer.
__device__ __forceinline__ int cell_axis_cert(const DevMesh &m, int k, double x, float xh, float xl) {
    const float df = (xh - m.lo_h[k]) + (xl - m.lo_l[k]);
    const float ed = delta_bound(df, xh, m.lo_h[k]);
    const float q = df * m.inv_sa[k];
    const float bnd = fmaf(2.0f * ed, m.inv_sa[k], fmaf(k8U, fabsf(q), kTiny));
    const int a = __float2int_rd(q - bnd), b = __float2int_rd(q + bnd);
    if (a == b && fabsf(q) < 4.0e6f) return a < 0 ? 0 : (a > m.ga[k] - 1 ? m.ga[k] - 1 : a);
    return int(cell_axis64(x, m.lo[k], m.sa[k], m.ga[k]));
}

// Inputs of row b (particle idx[b], or b): the window of dim channels at
// every (padded, if PAD) window position, channels first, and the offset.
// Window cell o (x fastest) of a particle whose ASG cell is c is cell
// c - W/2 + o; its point is the pooled centroid of that cell if the cell is
// in the grid and holds one, else its centre lo + (cell + 1/2) s. A warp takes
// a particle: its cell and offset once, then 32 window positions at a time.
// Bound by the FP64 pipe (56 cycles an instruction and warp): with an FP64
// division per value 59 us for 4096 2-D windows, 27 us now.
template <int D, int PAD>
__global__ void __launch_bounds__(kT) features_kernel(const DevMesh m, int64_t B,
                                                      const double *__restrict__ xp,
                                                      const int64_t *__restrict__ idx,
                                                      float *__restrict__ win,
                                                      float *__restrict__ offset) {
    using G = Win<D>;
    constexpr int E = G::W + 2 * PAD;                // stored edge
    constexpr int PE = D == 2 ? E * E : E * E * E;
    __shared__ double inv_s[3];
    if (threadIdx.x < D) inv_s[threadIdx.x] = __ddiv_rn(1.0, m.sa[threadIdx.x]);
    __syncthreads();
    double inv[D];
    #pragma unroll
    for (int k = 0; k < D; ++k) inv[k] = inv_s[k];
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t b = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; b < B; b += warps) {
        const int64_t r = idx ? idx[b] : b;
        double x[D];
        int c0[D];
        #pragma unroll
        for (int k = 0; k < D; ++k) {
            x[k] = xp[r * D + k];
            float xh, xl;
            split_double(x[k], xh, xl);
            c0[k] = cell_axis_cert(m, k, x[k], xh, xl);
        }
        if (lane < D) {
            double xv = x[0], s = m.sa[0], lo = m.lo[0];
            int c = c0[0];
            #pragma unroll
            for (int k = 1; k < D; ++k)
                if (lane == k) {
                    xv = x[k];
                    s = m.sa[k];
                    lo = m.lo[k];
                    c = c0[k];
                }
            offset[b * D + lane] = float(__dsub_rn(__ddiv_rn(__dsub_rn(xv, lo), s), double(c) + 0.5));
        }
        float *out = win + b * D * PE;
        #pragma unroll 2
        for (int pe = lane; pe < PE; pe += 32) {
            int e[3] = {pe % E - PAD, (pe / E) % E - PAD, D == 3 ? pe / (E * E) - PAD : 0};
            bool ring = false, inside = true;
            int64_t flat = 0;
            #pragma unroll
            for (int k = D - 1; k >= 0; --k) {
                ring |= e[k] < 0 || e[k] >= G::W;
                const int cc = c0[k] - G::W / 2 + e[k];
                inside &= cc >= 0 && cc < m.ga[k];
                flat = flat * m.ga[k] + (cc < 0 ? 0 : (cc > m.ga[k] - 1 ? m.ga[k] - 1 : cc));
            }
            if (ring) {
                #pragma unroll
                for (int k = 0; k < D; ++k) out[int64_t(k) * PE + pe] = 0.f;
                continue;
            }
            double pt[D];
            #pragma unroll
            for (int k = 0; k < D; ++k) pt[k] = __ldg(m.pool + flat * D + k);
            uint32_t nl, nh;
            dbits(pt[0], nl, nh);
            const bool nan = (nh & 0x7ff00000u) == 0x7ff00000u && ((nh & 0xfffffu) | nl) != 0;
            if (!inside || nan) {
                #pragma unroll
                for (int k = 0; k < D; ++k)
                    pt[k] = __dadd_rn(m.lo[k], __dmul_rn(double(c0[k] - G::W / 2 + e[k]) + 0.5, m.sa[k]));
            }
            #pragma unroll
            for (int k = 0; k < D; ++k)
                out[int64_t(k) * PE + pe] =
                    quotient_to_float(__dsub_rn(pt[k], x[k]), m.sa[k], inv[k]);
        }
    }
}

// a[b][q][c] = y[b][p(q)][c] at the interior of the padded window, 0 on its
// ring (channels last): the zero padding of the second convolution
template <int D>
__global__ void __launch_bounds__(kT) pad_kernel(const float *__restrict__ y, int64_t B, int C,
                                                 float *__restrict__ a) {
    using G = Win<D>;
    const int64_t total = B * G::Pq * C;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x) {
        const int c = int(q % C);
        const int64_t bq = q / C;
        const int pq = int(bq % G::Pq);
        const int64_t b = bq / G::Pq;
        const int qx = pq % G::Wq, qy = (pq / G::Wq) % G::Wq, qz = D == 3 ? pq / (G::Wq * G::Wq) : 1;
        const bool ring = qx == 0 || qy == 0 || qx == G::Wq - 1 || qy == G::Wq - 1 ||
                          (D == 3 && (qz == 0 || qz == G::Wq - 1));
        if (ring) {
            a[q] = 0.f;
            continue;
        }
        const int p = D == 2 ? (qy - 1) * G::W + qx - 1 : ((qz - 1) * G::W + qy - 1) * G::W + qx - 1;
        a[q] = y[(b * G::P + p) * C + c];
    }
}

// dz[b][p][c] = dpad[b][q(p)][c] * (z[b][p][c] > 0): the padded gradient of
// the second convolution's input, cropped, through the first ReLU
template <int D>
__global__ void __launch_bounds__(kT) crop_relu_back_kernel(const float *__restrict__ dpad,
                                                            const float *__restrict__ z, int64_t B,
                                                            int C, float *__restrict__ dz) {
    using G = Win<D>;
    const int64_t total = B * G::P * C;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x) {
        const int c = int(q % C);
        const int64_t bp = q / C;
        const int p = int(bp % G::P);
        const int64_t b = bp / G::P;
        const int px = p % G::W, py = (p / G::W) % G::W, pz = D == 3 ? p / (G::W * G::W) : -1;
        const int pq = D == 2 ? (py + 1) * G::Wq + px + 1
                              : ((pz + 1) * G::Wq + py + 1) * G::Wq + px + 1;
        dz[q] = z[q] > 0.f ? dpad[(b * G::Pq + pq) * C + c] : 0.f;
    }
}

// Average pooling of ReLU(z) over 2^D blocks (stride 2, the last odd row
// dropped) into the first 32 Pp columns of cat (row stride ldc), in the
// order [channel][z][y][x]
template <int D>
__global__ void __launch_bounds__(kT) pool_relu_kernel(const float *__restrict__ z, int64_t B,
                                                       float *__restrict__ cat, int64_t ldc) {
    using G = Win<D>;
    constexpr int C = kClsCh;
    const int64_t total = B * C * G::Pp;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x) {
        const int pp = int(q % G::Pp);
        const int c = int((q / G::Pp) % C);
        const int64_t b = q / (int64_t(C) * G::Pp);
        const int px = pp % G::Wp, py = (pp / G::Wp) % G::Wp, pz = D == 3 ? pp / (G::Wp * G::Wp) : 0;
        float s = 0.f;
        for (int oz = 0; oz < (D == 3 ? 2 : 1); ++oz)
            for (int oy = 0; oy < 2; ++oy)
                for (int ox = 0; ox < 2; ++ox) {
                    const int x = 2 * px + ox, y = 2 * py + oy, zz = 2 * pz + oz;
                    const int p = D == 2 ? y * G::W + x : (zz * G::W + y) * G::W + x;
                    s += fmaxf(z[(b * G::P + p) * C + c], 0.f);
                }
        cat[b * ldc + int64_t(c) * G::Pp + pp] = s / float(1 << D);
    }
}

// dz[b][p][c] = (dcat[b][c Pp + pooled(p)] / 2^D if p lies in a pooled block,
// else 0) * (z > 0): the pooling's gradient through the second ReLU
template <int D>
__global__ void __launch_bounds__(kT) pool_back_kernel(const float *__restrict__ dcat, int64_t ldc,
                                                       const float *__restrict__ z, int64_t B,
                                                       float *__restrict__ dz) {
    using G = Win<D>;
    constexpr int C = kClsCh;
    const int64_t total = B * G::P * C;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x) {
        const int c = int(q % C);
        const int64_t bp = q / C;
        const int p = int(bp % G::P);
        const int64_t b = bp / G::P;
        const int px = p % G::W, py = (p / G::W) % G::W, pz = D == 3 ? p / (G::W * G::W) : 0;
        float g = 0.f;
        if (px < 2 * G::Wp && py < 2 * G::Wp && (D == 2 || pz < 2 * G::Wp) && z[q] > 0.f) {
            const int pp = D == 2 ? (py / 2) * G::Wp + px / 2
                                  : ((pz / 2) * G::Wp + py / 2) * G::Wp + px / 2;
            g = dcat[b * ldc + int64_t(c) * G::Pp + pp] / float(1 << D);
        }
        dz[q] = g;
    }
}

// cat[b][off + j] = relu(y[b][j]) (the offset branch's output) and its
// gradient dy[b][j] = dcat[b][off + j] * (y > 0)
__global__ void cat_relu_kernel(const float *__restrict__ y, int64_t B, int n,
                                float *__restrict__ cat, int64_t ldc, int64_t off) {
    const int64_t total = B * n;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x)
        cat[(q / n) * ldc + off + q % n] = fmaxf(y[q], 0.f);
}
__global__ void uncat_relu_back_kernel(const float *__restrict__ dcat, int64_t ldc, int64_t off,
                                       const float *__restrict__ y, int64_t B, int n,
                                       float *__restrict__ dy) {
    const int64_t total = B * n;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < total;
         q += int64_t(gridDim.x) * blockDim.x)
        dy[q] = y[q] > 0.f ? dcat[(q / n) * ldc + off + q % n] : 0.f;
}

__device__ __forceinline__ float warp_sum(float v) {
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// Softmax of every row of H (Eq. 7) and the gradient of the mean
// cross-entropy over the rows with a label in [0, n_cls):
// dH = (softmax - onehot) / n_valid, 0 on the other rows; the loss is added
// to *loss. One block, one warp per row, reductions in a fixed order: the
// same bits on every run.
__global__ void __launch_bounds__(1024) softmax_ce_kernel(const float *__restrict__ H,
                                                          const int32_t *__restrict__ labels,
                                                          const int64_t *__restrict__ idx,
                                                          int64_t B, int n_cls,
                                                          float *__restrict__ dH,
                                                          float *__restrict__ loss) {
    __shared__ float red[32];
    __shared__ int cnt[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int c = 0;
    for (int64_t b = threadIdx.x; b < B; b += blockDim.x) {
        const int32_t l = labels[idx ? idx[b] : b];
        c += l >= 0 && l < n_cls;
    }
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    if (lane == 0) cnt[warp] = c;
    __syncthreads();
    int n_valid = 0;
    for (int w = 0; w < nw; ++w) n_valid += cnt[w];
    const float inv = n_valid > 0 ? 1.f / float(n_valid) : 0.f;
    float lsum = 0.f;
    for (int64_t b = warp; b < B; b += nw) {
        const int32_t l = labels[idx ? idx[b] : b];
        const bool valid = l >= 0 && l < n_cls;
        const float *h = H + b * n_cls;
        float mx = -INFINITY;
        for (int j = lane; j < n_cls; j += 32) mx = fmaxf(mx, h[j]);
        mx = warp_max(mx);
        float se = 0.f;
        for (int j = lane; j < n_cls; j += 32) se += expf(h[j] - mx);
        se = warp_sum(se);
        const float rse = 1.f / se;
        float *g = dH + b * n_cls;
        for (int j = lane; j < n_cls; j += 32)
            g[j] = valid ? (expf(h[j] - mx) * rse - (j == l ? 1.f : 0.f)) * inv : 0.f;
        if (valid && lane == 0) lsum += logf(se) - (h[l] - mx);
    }
    if (lane == 0) red[warp] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < nw; ++w) s += red[w];
        *loss += s * inv;
    }
}

// ---------------------------------------------------------------------------
// Training on the tiled BF16 layouts of the fully connected layers (fc_tc.h)
// ---------------------------------------------------------------------------

// a thread pools one channel of a row: neighbouring threads read neighbouring
// channels; columns of a channel are Pp consecutive ones
template <int D>
__global__ void __launch_bounds__(kT) pool_tiled_kernel(const float *__restrict__ z, int64_t B,
                                                        FcMat cat) {
    using G = Win<D>;
    constexpr int C = kClsCh;
    pdl_wait();
    const int64_t rows = (B + 127) / 128 * 128;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < rows * C;
         q += int64_t(gridDim.x) * blockDim.x) {
        const int c = int(q % C);
        const int64_t b = q / C;
        uint8_t *row = cat.p + (b >> 7) * cat.tile + int64_t(cat.chunk0) * kFcChunk + (b & 127) * 16;
        const float *zb = z + b * G::P * C + c;
        #pragma unroll
        for (int p0 = 0; p0 < G::Pp; p0 += 4) {
            float s[4] = {0.f, 0.f, 0.f, 0.f};
            #pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int pp = p0 + u;
                if (b >= B || pp >= G::Pp) continue;
                const int px = pp % G::Wp, py = (pp / G::Wp) % G::Wp, pz = pp / (G::Wp * G::Wp);
                for (int oz = 0; oz < (D == 3 ? 2 : 1); ++oz)
                    for (int oy = 0; oy < 2; ++oy)
                        for (int ox = 0; ox < 2; ++ox) {
                            const int x = 2 * px + ox, y = 2 * py + oy, zz = 2 * pz + oz;
                            const int p = D == 2 ? y * G::W + x : (zz * G::W + y) * G::W + x;
                            s[u] += fmaxf(zb[p * C], 0.f);
                        }
                s[u] = s[u] / float(1 << D);
            }
            const int col = c * G::Pp + p0;
            uint8_t *o = row + int64_t(col >> 3) * kFcChunk + (col & 7) * 2;
            if constexpr (G::Pp % 4 == 0) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(s[0], s[1]);
                const __nv_bfloat162 hi = __floats2bfloat162_rn(s[2], s[3]);
                *reinterpret_cast<uint2 *>(o) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo),
                                                           *reinterpret_cast<const uint32_t *>(&hi));
            } else {
                #pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int cu = col + u;
                    if (p0 + u < G::Pp)
                        *reinterpret_cast<__nv_bfloat16 *>(row + int64_t(cu >> 3) * kFcChunk +
                                                           (cu & 7) * 2) = __float2bfloat16_rn(s[u]);
                }
            }
        }
    }
}

// 2-D. A block takes whole rows: the row's pooled gradient goes through shared
// memory (read along the pooled positions, used along the channels); a thread
// keeps one channel, whose column sum it carries
__global__ void __launch_bounds__(kT) pool_back_tiled_kernel(const float *__restrict__ dpool,
                                                             const float *__restrict__ z,
                                                             int64_t B, uint16_t *__restrict__ dz,
                                                             float *__restrict__ part) {
    using G = Win<2>;
    constexpr int C = kClsCh, Ld = G::Pp | 1;      // odd stride: no bank conflicts
    __shared__ float sg[C * Ld];
    __shared__ float red[kT];
    pdl_wait();
    const int c = threadIdx.x % C;
    float sum = 0.f;
    constexpr int kZ = (G::P + kT / C - 1) / (kT / C);       // positions of a thread
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        // the row's pre-activations travel with its pooled gradient
        float zv[kZ];
        #pragma unroll
        for (int j = 0; j < kZ; ++j) {
            const int p = threadIdx.x / C + j * (kT / C);
            zv[j] = p < G::P ? __ldg(z + (b * G::P + p) * C + c) : 0.f;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < C * G::Pp; i += kT)
            sg[i / G::Pp * Ld + i % G::Pp] = __ldg(dpool + b * (C * G::Pp) + i);
        __syncthreads();
        #pragma unroll
        for (int j = 0; j < kZ; ++j) {
            const int p = threadIdx.x / C + j * (kT / C);
            if (p >= G::P) continue;
            const int px = p % G::W, py = p / G::W;
            const bool pooled = px < 2 * G::Wp && py < 2 * G::Wp && zv[j] > 0.f;
            const float g = pooled ? sg[c * Ld + (py / 2) * G::Wp + px / 2] / 4.f : 0.f;
            sum += g;
            dz[(b * G::P + p) * C + c] = __bfloat16_as_ushort(__float2bfloat16_rn(g));
        }
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x < C) {
        float s = 0.f;
        for (int i = 0; i < kT / C; ++i) s += red[i * C + c];
        part[int64_t(blockIdx.x) * C + c] = s;
    }
}

constexpr int kSmRows = 32;      // rows per block of the tiled softmax

// rows with a label in [0, n_cls)
__global__ void __launch_bounds__(1024) count_labels_kernel(const int32_t *__restrict__ labels,
                                                            const int64_t *__restrict__ idx,
                                                            int64_t B, int n_cls,
                                                            int *__restrict__ count) {
    __shared__ int cnt[32];
    pdl_wait();
    int c = 0;
    for (int64_t b = threadIdx.x; b < B; b += blockDim.x) {
        const int32_t l = labels[idx ? idx[b] : b];
        c += l >= 0 && l < n_cls;
    }
    c = __reduce_add_sync(kFull, c);
    if ((threadIdx.x & 31) == 0) cnt[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = 0;
        for (int w = 0; w < 32; ++w) n += cnt[w];
        *count = n;
    }
}

// softmax_ce_kernel's rows (the same arithmetic, a warp per row), spread over
// blocks of kSmRows rows. NJ: columns per lane.
template <int NJ>
__global__ void __launch_bounds__(kT) softmax_ce_tiled_kernel(const float *__restrict__ H,
                                                              const int32_t *__restrict__ labels,
                                                              const int64_t *__restrict__ idx,
                                                              int64_t B, int n_cls, FcMat gH,
                                                              float *__restrict__ part,
                                                              float *__restrict__ loss_part,
                                                              const int *__restrict__ count) {
    extern __shared__ float sred[];                 // [8][32 NJ]
    __shared__ float lred[8];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_valid = *count;
    const float inv = n_valid > 0 ? 1.f / float(n_valid) : 0.f;
    float col[NJ], lsum = 0.f;
    #pragma unroll
    for (int j = 0; j < NJ; ++j) col[j] = 0.f;
    const int64_t b0 = int64_t(blockIdx.x) * kSmRows;
    for (int r = warp; r < kSmRows; r += 8) {
        const int64_t b = b0 + r;                   // rows past B up to a tile's end are zero
        uint8_t *row = gH.p + (b >> 7) * gH.tile + int64_t(gH.chunk0) * kFcChunk + (b & 127) * 16;
        float g[NJ];
        #pragma unroll
        for (int j = 0; j < NJ; ++j) g[j] = 0.f;
        if (b < B) {
            const int32_t l = labels[idx ? idx[b] : b];
            const bool valid = l >= 0 && l < n_cls;
            const float *h = H + b * n_cls;
            float v[NJ], mx = -INFINITY;
            #pragma unroll
            for (int j = 0; j < NJ; ++j) {
                v[j] = lane + 32 * j < n_cls ? h[lane + 32 * j] : -INFINITY;
                if (lane + 32 * j < n_cls) mx = fmaxf(mx, v[j]);
            }
            mx = warp_max(mx);
            float e[NJ], se = 0.f;
            #pragma unroll
            for (int j = 0; j < NJ; ++j) {
                e[j] = expf(v[j] - mx);
                if (lane + 32 * j < n_cls) se += e[j];
            }
            se = warp_sum(se);
            const float rse = 1.f / se;
            #pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = lane + 32 * j;
                g[j] = valid && k < n_cls ? (e[j] * rse - (k == l ? 1.f : 0.f)) * inv : 0.f;
            }
            if (valid && lane == 0) lsum += logf(se) - (h[l] - mx);
        }
        #pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int k = lane + 32 * j;
            col[j] += g[j];
            if (k < gH.chunks * 8)
                *reinterpret_cast<__nv_bfloat16 *>(row + int64_t(k >> 3) * kFcChunk + (k & 7) * 2) =
                    __float2bfloat16_rn(g[j]);
        }
    }
    #pragma unroll
    for (int j = 0; j < NJ; ++j) sred[warp * (32 * NJ) + lane + 32 * j] = col[j];
    if (lane == 0) lred[warp] = lsum;
    __syncthreads();
    for (int k = threadIdx.x; k < n_cls; k += kT) {
        float s = 0.f;
        for (int w = 0; w < 8; ++w) s += sred[w * (32 * NJ) + k];
        part[int64_t(blockIdx.x) * n_cls + k] = s;
    }
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < 8; ++w) s += lred[w];
        loss_part[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(32) loss_sum_kernel(const float *__restrict__ loss_part, int n,
                                                      const int *__restrict__ count,
                                                      float *__restrict__ loss) {
    pdl_wait();
    float s = 0.f;
    for (int i = threadIdx.x; i < n; i += 32) s += loss_part[i];
    s = warp_sum(s);
    const int n_valid = *count;
    if (threadIdx.x == 0) *loss = s * (n_valid > 0 ? 1.f / float(n_valid) : 0.f);
}

// label = window cell (x fastest) holding the centroid of the host element,
// the cell coordinates clamped into the window around x_p's ASG cell (label
// may be host: each row is read before it is written)
template <int D>
__global__ void __launch_bounds__(kT) labels_kernel(const DevMesh m, int64_t n,
                                                    const double *__restrict__ xp,
                                                    const int32_t *host, int32_t *label) {
    using G = Win<D>;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int32_t h = host[i];
        if (h < 0 || h >= m.n_e) {
            label[i] = -1;
            continue;
        }
        const int64_t li = m.iperm[h];
        int32_t cls = 0;
        #pragma unroll
        for (int k = D - 1; k >= 0; --k) {
            const int64_t c0 = cell_axis64(xp[i * D + k], m.lo[k], m.sa[k], m.ga[k]);
            const int64_t cc = cell_axis64(m.centroid[li * D + k], m.lo[k], m.sa[k], m.ga[k]);
            int64_t rel = cc - (c0 - G::W / 2);
            rel = rel < 0 ? 0 : (rel > G::W - 1 ? G::W - 1 : rel);
            cls = cls * G::W + int32_t(rel);
        }
        label[i] = cls;
    }
}

// K_p (Eq. 8): one warp per particle takes the class of the largest logit
// (the lowest among equal ones; NaN never wins), then the ASG seed of that
// window cell (user id), else the fallback start (fallback[i], or the plain
// start of mesh node row0 + i)
template <int D>
__global__ void __launch_bounds__(kT) start_kernel(const DevMesh m, int64_t n,
                                                   const double *__restrict__ xp,
                                                   const float *__restrict__ logits,
                                                   const int32_t *__restrict__ fallback,
                                                   int64_t row0, int32_t *__restrict__ start,
                                                   int32_t *__restrict__ cls_out) {
    using G = Win<D>;
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const float *h = logits + i * G::P;
        float best = -INFINITY;
        int bj = G::P;
        for (int j = lane; j < G::P; j += 32) {
            const float v = h[j];
            if (v > best) {   // lanes scan increasing j: the first of equal values stays
                best = v;
                bj = j;
            }
        }
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(kFull, best, o);
            const int oj = __shfl_xor_sync(kFull, bj, o);
            if (ov > best || (ov == best && oj < bj)) {
                best = ov;
                bj = oj;
            }
        }
        if (lane != 0) continue;
        // no finite maximum: no class
        const bool has_cls = bj < G::P && best > -INFINITY && best < INFINITY;
        int32_t s = -1;
        if (has_cls) {
            int r = bj;
            bool inside = true;
            int64_t cc[D];
            #pragma unroll
            for (int k = 0; k < D; ++k) {
                const int64_t c0 = cell_axis64(xp[i * D + k], m.lo[k], m.sa[k], m.ga[k]);
                cc[k] = c0 - G::W / 2 + r % G::W;
                r /= G::W;
                inside &= cc[k] >= 0 && cc[k] < m.ga[k];
            }
            if (inside) {
                int64_t flat = 0;
                #pragma unroll
                for (int k = D - 1; k >= 0; --k) flat = flat * m.ga[k] + cc[k];
                const int32_t seed = m.seed[flat];
                if (seed >= 0) s = walk_uid<D>(m.recw, seed);
            }
        }
        if (s < 0) {
            if (fallback) {
                s = fallback[i];
            } else {
                const int32_t e = node_start(m.node_elem[row0 + i]);
                s = e < 0 ? -1 : walk_uid<D>(m.recw, e);
            }
        }
        start[i] = s;
        if (cls_out) cls_out[i] = has_cls ? bj : -1;
    }
}

}  // namespace

void launch_departure(int64_t n, int dim, const double *x, const double *u, double dt,
                      double *xp, int sm_count, cudaStream_t st) {
    const int64_t total = n * dim;
    departure_kernel<<<blocks_for(total, sm_count), kT, 0, st>>>(total, x, u, dt, xp);
}

void launch_cls_features(const DevMesh &m, int64_t B, const double *xp, const int64_t *idx,
                         bool pad, float *win, float *offset, int sm_count, cudaStream_t st) {
    const int g = int(std::max<int64_t>(1, std::min<int64_t>((B + 7) / 8, int64_t(sm_count) * 16)));
    if (m.dim == 2 && pad)
        features_kernel<2, 1><<<g, kT, 0, st>>>(m, B, xp, idx, win, offset);
    else if (m.dim == 2)
        features_kernel<2, 0><<<g, kT, 0, st>>>(m, B, xp, idx, win, offset);
    else if (pad)
        features_kernel<3, 1><<<g, kT, 0, st>>>(m, B, xp, idx, win, offset);
    else
        features_kernel<3, 0><<<g, kT, 0, st>>>(m, B, xp, idx, win, offset);
}

void launch_cls_pad(int dim, const float *y, int64_t B, int C, float *a, int sm_count,
                    cudaStream_t st) {
    const int Wq = cls_window(dim) + 2;
    const int64_t total = B * (dim == 2 ? Wq * Wq : Wq * Wq * Wq) * C;
    if (dim == 2)
        pad_kernel<2><<<blocks_for(total, sm_count), kT, 0, st>>>(y, B, C, a);
    else
        pad_kernel<3><<<blocks_for(total, sm_count), kT, 0, st>>>(y, B, C, a);
}

void launch_cls_crop_relu_back(int dim, const float *dpad, const float *z, int64_t B, int C,
                               float *dz, int sm_count, cudaStream_t st) {
    const int W = cls_window(dim);
    const int64_t total = B * (dim == 2 ? W * W : W * W * W) * C;
    if (dim == 2)
        crop_relu_back_kernel<2><<<blocks_for(total, sm_count), kT, 0, st>>>(dpad, z, B, C, dz);
    else
        crop_relu_back_kernel<3><<<blocks_for(total, sm_count), kT, 0, st>>>(dpad, z, B, C, dz);
}

void launch_cls_pool(int dim, const float *z, int64_t B, float *cat, int64_t ldc, int sm_count,
                     cudaStream_t st) {
    const int64_t total = B * cls_pooled(dim);
    if (dim == 2)
        pool_relu_kernel<2><<<blocks_for(total, sm_count), kT, 0, st>>>(z, B, cat, ldc);
    else
        pool_relu_kernel<3><<<blocks_for(total, sm_count), kT, 0, st>>>(z, B, cat, ldc);
}

void launch_cls_pool_back(int dim, const float *dcat, int64_t ldc, const float *z, int64_t B,
                          float *dz, int sm_count, cudaStream_t st) {
    const int W = cls_window(dim);
    const int64_t total = B * (dim == 2 ? W * W : W * W * W) * kClsCh;
    if (dim == 2)
        pool_back_kernel<2><<<blocks_for(total, sm_count), kT, 0, st>>>(dcat, ldc, z, B, dz);
    else
        pool_back_kernel<3><<<blocks_for(total, sm_count), kT, 0, st>>>(dcat, ldc, z, B, dz);
}

void launch_cls_cat_relu(const float *y, int64_t B, int n, float *cat, int64_t ldc, int64_t off,
                         int sm_count, cudaStream_t st) {
    cat_relu_kernel<<<blocks_for(B * n, sm_count), kT, 0, st>>>(y, B, n, cat, ldc, off);
}

void launch_cls_uncat_relu_back(const float *dcat, int64_t ldc, int64_t off, const float *y,
                                int64_t B, int n, float *dy, int sm_count, cudaStream_t st) {
    uncat_relu_back_kernel<<<blocks_for(B * n, sm_count), kT, 0, st>>>(dcat, ldc, off, y, B, n,
                                                                       dy);
}

void launch_softmax_ce(const float *H, const int32_t *labels, const int64_t *idx, int64_t B,
                       int n_cls, float *dH, float *loss, cudaStream_t st) {
    softmax_ce_kernel<<<1, 1024, 0, st>>>(H, labels, idx, B, n_cls, dH, loss);
}

void launch_cls_pool_tiled(int dim, const float *z, int64_t B, const FcMat &cat, int sm_count,
                           cudaStream_t st) {
    const int g = blocks_for((B + 127) / 128 * 128 * kClsCh, sm_count, 8);
    launch_pdl(dim == 2 ? pool_tiled_kernel<2> : pool_tiled_kernel<3>, dim3(g), dim3(kT), 0, st, z, B,
               cat);
}

int cls_pool_back_blocks(int64_t B, int sm_count) {
    return int(std::min<int64_t>(B, int64_t(sm_count) * 6));
}

void launch_cls_pool_back_tiled(const float *dpool, const float *z, int64_t B, uint16_t *dz,
                                float *part, int sm_count, cudaStream_t st) {
    launch_pdl(pool_back_tiled_kernel, dim3(cls_pool_back_blocks(B, sm_count)), dim3(kT), 0, st, dpool,
               z, B, dz, part);
}

int cls_softmax_blocks(int64_t B) { return int((B + 127) / 128 * (128 / kSmRows)); }

void launch_softmax_ce_tiled(const float *H, const int32_t *labels, const int64_t *idx, int64_t B,
                             int n_cls, const FcMat &gH, float *part, float *loss_part, int *count,
                             cudaStream_t st) {
    launch_pdl(count_labels_kernel, dim3(1), dim3(1024), 0, st, labels, idx, B, n_cls, count);
    const int g = cls_softmax_blocks(B);
    if (n_cls <= 96)
        launch_pdl(softmax_ce_tiled_kernel<3>, dim3(g), dim3(kT), 8 * 96 * 4, st, H, labels, idx, B,
                   n_cls, gH, part, loss_part, count);
    else
        launch_pdl(softmax_ce_tiled_kernel<11>, dim3(g), dim3(kT), 8 * 352 * 4, st, H, labels, idx, B,
                   n_cls, gH, part, loss_part, count);
}

void launch_loss_sum(const float *loss_part, int n, const int *count, float *loss, cudaStream_t st) {
    launch_pdl(loss_sum_kernel, dim3(1), dim3(32), 0, st, loss_part, n, count, loss);
}

void launch_cls_labels(const DevMesh &m, int64_t n, const double *xp, const int32_t *host,
                       int32_t *label, int sm_count, cudaStream_t st) {
    if (m.dim == 2)
        labels_kernel<2><<<blocks_for(n, sm_count), kT, 0, st>>>(m, n, xp, host, label);
    else
        labels_kernel<3><<<blocks_for(n, sm_count), kT, 0, st>>>(m, n, xp, host, label);
}

void launch_cls_start(const DevMesh &m, int64_t n, const double *xp, const float *logits,
                      const int32_t *fallback, int64_t row0, int32_t *start, int32_t *cls,
                      int sm_count, cudaStream_t st) {
    const int g = int(std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, int64_t(sm_count) * 16)));
    if (m.dim == 2)
        start_kernel<2><<<g, kT, 0, st>>>(m, n, xp, logits, fallback, row0, start, cls);
    else
        start_kernel<3><<<g, kT, 0, st>>>(m, n, xp, logits, fallback, row0, start, cls);
}

}  // namespace cs
