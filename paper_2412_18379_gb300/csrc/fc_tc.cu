// Fully connected layers on the tensor cores with BF16 operands that never
// change layout: activations live in global memory as row tiles of 128 in the
// MMA's own operand order ([K / 8][128][8]), weights are packed the same way,
// so a pipeline stage is two contiguous blocks fetched by one bulk
// asynchronous copy each (no tensor map, no staging by threads), and an
// epilogue's warp stores 512 contiguous bytes per 8 columns. Read with the
// transposed descriptor the same tiles are the operands of the weight
// gradients (K = row).
//
// fc_gemm: one producer thread, one MMA-issuing warp, eight epilogue warps;
// four stages of K = 64; two accumulators, so the epilogue of a tile (bias,
// ReLU or its gate, BF16, column sums) runs under the next tile's products.
// The sums run in K order in K = 16 steps, as the general GEMM's
// (tc_gemm.cu), which staged FP32 operands through the threads and needed a
// separate pass for every bias, ReLU and layout change.
//
// Bound by the copies' latency and the epilogues (these layers' K is short), not
// by the tensor pipe. A chunk of 32768 particles in 2-D: xp2 11 us, fusion 26 us,
// logits 15 us; with four epilogue warps and the bias read from global memory 25,
// 48 and 20 us. A forward pass of 160801 particles took 3016 us with these layers
// on the general GEMM, 1420 us with them here and module 1 as it was.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "fc_tc.h"
#include "tc_common.cuh"

namespace cs {
namespace {

constexpr int kFcEpi = 8;            // epilogue warps: two per TMEM lane quarter
constexpr int kFcThreads = (2 + kFcEpi) * 32;   // producer, MMA, epilogue
constexpr int kFcBiasMax = 512;
constexpr int kStages = 4, kStageChunks = 8;
constexpr int kCh = int(kFcChunk);   // bytes of one 8-column chunk of a row tile

// bulk copy of contiguous global memory to shared memory, completing on `bar`
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// bounded wait for a phase, at a kernel's end (no abort flag, nothing raised)
__device__ __forceinline__ void settle(uint64_t *bar, uint32_t parity) {
    for (uint32_t i = 0; i < (1u << 24) && !mbar_try_wait(bar, parity); ++i)
        if (i > 64) __nanosleep(64);
}

struct FcArgs {
    FcMat A, gate, out;
    const uint8_t *B;
    int64_t M;
    int mt, nt, chunks, N;
    const float *bias;
    int relu;
    float *f32;
    int64_t ldf;
    float *colsum;
    int nsplit, split_stages;     // stages (of 64 columns) per split
    uint32_t cols;                // TMEM columns allocated
};

template <int BN>
struct FcGeo {
    static_assert(BN % 16 == 0 && BN <= 256, "MMA N");
    static constexpr int kA = kStageChunks * kCh;
    static constexpr int kB = kStageChunks * BN * 16;
    static constexpr int kStage = kA + kB;
    static constexpr int kTile = kStages * kStage;                  // f32 [kFcEpi][32 * 17]
    static constexpr int kBias = kTile + kFcEpi * 32 * 17 * 4;      // f32 [kFcBiasMax]
    static constexpr int kBar = kBias + kFcBiasMax * 4;             // full, empty, tfull, tempty
    static constexpr int kSlot = kBar + (2 * kStages + 5) * 8;
    static constexpr int kTotal = kSlot + 16;
    static_assert(kTotal <= 232448 && kStage % 128 == 0, "shared memory of one CTA");
};

template <int BN>
__global__ void __launch_bounds__(kFcThreads, 1) fc_gemm_kernel(const FcArgs a, int *err) {
    using G = FcGeo<BN>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + G::kBar), *empty = full + kStages;
    uint64_t *tfull = empty + kStages, *tempty = tfull + 2, *last = tempty + 2;
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + G::kSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + G::kSlot + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full + i, 1u);
            mbar_init(empty + i, 1u);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull + i, 1u);
            mbar_init(tempty + i, uint32_t(kFcEpi));
        }
        mbar_init(last, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(slot)),
                     "r"(a.cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    pdl_wait();
    const uint32_t tmem = *slot;
    // two accumulators alternate between tiles; a split sum takes nsplit side
    // by side and has one set
    const uint32_t nbuf = a.nsplit > 1 ? 1u : 2u;
    const int tiles = a.mt * a.nt, nst = (a.chunks + kStageChunks - 1) / kStageChunks;
    if (warp == 0) {
        if (elect_one()) {
            uint32_t s = 0, it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                const int m = t / a.nt, n = t % a.nt;
                const uint8_t *A = a.A.p + m * a.A.tile + int64_t(a.A.chunk0) * kCh;
                const uint8_t *B = a.B + int64_t(n) * a.chunks * (BN * 16);
                for (int j = 0; j < nst; ++j, ++it) {
                    s = it % kStages;
                    if (it >= kStages)
                        ok = mbar_wait(empty + s, (it / kStages - 1) & 1u, abort_flag, err);
                    if (!ok) break;
                    const int nc = min(kStageChunks, a.chunks - j * kStageChunks);
                    uint8_t *d = smem + s * G::kStage;
                    expect_tx(full + s, uint32_t(nc * (kCh + BN * 16)));
                    bulk_load(d, A + int64_t(j) * kStageChunks * kCh, uint32_t(nc * kCh), full + s);
                    bulk_load(d + G::kA, B + int64_t(j) * kStageChunks * BN * 16,
                              uint32_t(nc * BN * 16), full + s);
                }
            }
            // no copy of this CTA is in flight past this point
            for (uint32_t i = it > kStages ? it - kStages : 0; i < it; ++i)
                settle(full + i % kStages, (i / kStages) & 1u);
        }
        __syncwarp();
    } else if (warp == 1) {
        const bool leader = elect_one();
        constexpr uint32_t id = idesc_bf16(128, BN);
        uint32_t it = 0, i = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++i) {
            const uint32_t buf = i % nbuf;
            if (i >= nbuf) ok = warp_wait(tempty + buf, (i / nbuf - 1) & 1u, abort_flag, err);
            if (!ok) break;
            fence_after();
            for (int j = 0; j < nst; ++j, ++it) {
                const uint32_t s = it % kStages;
                ok = warp_wait(full + s, (it / kStages) & 1u, abort_flag, err);
                if (!ok) break;
                fence_after();
                if (leader) {
                    const uint32_t base = smem_addr(smem + s * G::kStage);
                    const uint64_t da = sdesc(base, kCh, 128), db = sdesc(base + G::kA, BN * 16, 128);
                    const int nq = min(kStageChunks, a.chunks - j * kStageChunks) / 2;
                    const int sp = a.nsplit > 1 ? j / a.split_stages : 0;
                    const int j0 = sp * a.split_stages;
                    const uint32_t d = tmem + buf * (a.cols / 2) + uint32_t(sp * BN);
                    for (int q = 0; q < nq; ++q)
                        mma_bf16(d, da + uint64_t(2 * q * (kCh >> 4)), db + uint64_t(2 * q * BN), id,
                                 j > j0 || q > 0 ? 1u : 0u);
                    mma_commit(empty + s);
                    if (j + 1 == nst) mma_commit(tfull + buf);
                }
                __syncwarp();
            }
        }
        if (leader) {
            mma_commit(last);
            settle(last, 0);
        }
        __syncwarp();
    } else {
        // warps w and w + 4 share a lane quarter and take alternate 16-column pieces
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        float *tile = reinterpret_cast<float *>(smem + G::kTile) + (warp - 2) * (32 * 17);
        float *bias = reinterpret_cast<float *>(smem + G::kBias);
        if (a.bias) {
            for (int j = tid - 64; j < a.N; j += kFcEpi * 32) bias[j] = __ldg(a.bias + j);
            asm volatile("bar.sync 1, %0;" ::"n"(kFcEpi * 32) : "memory");
        }
        uint32_t i = 0;
        for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++i) {
            const uint32_t buf = i % nbuf;
            if (!warp_wait(tfull + buf, (i / nbuf) & 1u, abort_flag, err)) break;
            fence_after();
            const int m = t / a.nt, n0 = (t % a.nt) * BN;
            const int r = 32 * quarter + lane;
            const int64_t row = int64_t(m) * 128 + r;
            const bool in = row < a.M;
            const uint32_t tq = tmem + buf * (a.cols / 2) + (uint32_t(32 * quarter) << 16);
            #pragma unroll 1
            for (int c = 16 * half; c < BN; c += 32) {
                if (n0 + c >= a.N) break;
                float v[16];
                tmem_ld16(tq + uint32_t(c), v);
                for (int sp = 1; sp < a.nsplit; ++sp) {
                    float u[16];
                    tmem_ld16(tq + uint32_t(sp * BN + c), u);
                    #pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] += u[e];
                }
                if (a.bias) {
                    #pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float4 b = *reinterpret_cast<const float4 *>(bias + n0 + c + 4 * e);
                        v[4 * e] += b.x;
                        v[4 * e + 1] += b.y;
                        v[4 * e + 2] += b.z;
                        v[4 * e + 3] += b.w;
                    }
                }
                if (a.relu) {
                    #pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = fmaxf(v[e], 0.f);
                }
                if (a.gate.p) {
                    const uint8_t *g = a.gate.p + m * a.gate.tile +
                                       int64_t(a.gate.chunk0 + (n0 + c) / 8) * kCh + r * 16;
                    #pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint4 w = __ldg(reinterpret_cast<const uint4 *>(g + h * kCh));
                        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                        #pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const uint32_t b = (ww[e >> 1] >> (16 * (e & 1))) & 0xffffu;
                            v[8 * h + e] = b != 0 && b < 0x8000u ? v[8 * h + e] : 0.f;
                        }
                    }
                }
                if (!in) {
                    #pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = 0.f;
                }
                if (a.out.p) {
                    uint8_t *o = a.out.p + m * a.out.tile +
                                 int64_t(a.out.chunk0 + (n0 + c) / 8) * kCh + r * 16;
                    uint32_t h[8];
                    #pragma unroll
                    for (int e = 0; e < 8; ++e) h[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
                    *reinterpret_cast<uint4 *>(o) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4 *>(o + kCh) = make_uint4(h[4], h[5], h[6], h[7]);
                }
                if (a.f32 || a.colsum) {
                    #pragma unroll
                    for (int e = 0; e < 16; ++e) tile[lane * 17 + e] = v[e];
                    __syncwarp();
                    const int e = lane & 15, col = n0 + c + e;
                    if (a.f32 && col < a.N) {
                        // 16 consecutive floats of two rows per store
                        #pragma unroll 4
                        for (int q = lane >> 4; q < 32; q += 2) {
                            const int64_t ii = int64_t(m) * 128 + 32 * quarter + q;
                            if (ii < a.M) a.f32[ii * a.ldf + col] = tile[q * 17 + e];
                        }
                    }
                    if (a.colsum) {
                        float s = 0.f;
                        #pragma unroll
                        for (int q = 0; q < 16; ++q) s += tile[(16 * (lane >> 4) + q) * 17 + e];
                        s += __shfl_xor_sync(kFull, s, 16);
                        if (lane < 16 && col < a.N) a.colsum[(int64_t(m) * 4 + quarter) * a.N + col] = s;
                    }
                    __syncwarp();
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty + buf);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.cols));
}

// Weight gradients: one CTA per (128 n, 256 k, split of the row tiles); a
// stage is one row tile of both operands (K = 128 rows, 8 MMAs of N = 256).
struct FcWgArgs {
    FcMat Y, X;
    int64_t row_tiles;
    int N, K, per;                // per: row tiles of a split
    float *part;
};
struct FcWgGeo {
    static constexpr int BK = 256;
    static constexpr int kY = 16 * kCh, kX = (BK / 8) * kCh, kStage = kY + kX;
    static constexpr int kStagesW = 2;
    static constexpr int kTile = kStagesW * kStage;
    static constexpr int kBar = kTile + kFcEpi * 32 * 17 * 4;
    static constexpr int kSlot = kBar + 8 * (2 * kStagesW + 1);
    static constexpr int kTotal = kSlot + 16;
    static_assert(kTotal <= 232448, "shared memory of one CTA");
};

__global__ void __launch_bounds__(kFcThreads, 1) fc_wgrad_kernel(const FcWgArgs a, int *err) {
    using G = FcWgGeo;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + G::kBar), *empty = full + G::kStagesW;
    uint64_t *done = empty + G::kStagesW;
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + G::kSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + G::kSlot + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < G::kStagesW; ++i) {
            mbar_init(full + i, 1u);
            mbar_init(empty + i, 1u);
        }
        mbar_init(done, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(
            smem_addr(slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    pdl_wait();
    const uint32_t tmem = *slot;
    const int n0 = blockIdx.x * 128, k0 = blockIdx.y * G::BK;
    const int64_t t0 = int64_t(blockIdx.z) * a.per, t1 = min(a.row_tiles, t0 + a.per);
    // chunks of this CTA's operands that exist (the rest of a stage is never
    // written; it only feeds rows and columns that are not stored)
    const int yc = min(16, a.Y.chunks - n0 / 8), xc = min(G::BK / 8, a.X.chunks - k0 / 8);
    if (warp == 0) {
        if (elect_one()) {
            uint32_t it = 0;
            for (int64_t t = t0; t < t1; ++t, ++it) {
                const uint32_t s = it % G::kStagesW;
                if (it >= G::kStagesW &&
                    !mbar_wait(empty + s, (it / G::kStagesW - 1) & 1u, abort_flag, err))
                    break;
                uint8_t *d = smem + s * G::kStage;
                expect_tx(full + s, uint32_t((yc + xc) * kCh));
                bulk_load(d, a.Y.p + t * a.Y.tile + int64_t(a.Y.chunk0 + n0 / 8) * kCh,
                          uint32_t(yc * kCh), full + s);
                bulk_load(d + G::kY, a.X.p + t * a.X.tile + int64_t(a.X.chunk0 + k0 / 8) * kCh,
                          uint32_t(xc * kCh), full + s);
            }
            for (uint32_t i = it > G::kStagesW ? it - G::kStagesW : 0; i < it; ++i)
                settle(full + i % G::kStagesW, (i / G::kStagesW) & 1u);
        }
        __syncwarp();
    } else if (warp == 1) {
        const bool leader = elect_one();
        constexpr uint32_t id = idesc_mn(idesc_bf16(128, G::BK), true, true);
        uint32_t it = 0;
        bool ok = true;
        for (int64_t t = t0; t < t1 && ok; ++t, ++it) {
            const uint32_t s = it % G::kStagesW;
            ok = warp_wait(full + s, (it / G::kStagesW) & 1u, abort_flag, err);
            if (!ok) break;
            fence_after();
            if (leader) {
                const uint32_t base = smem_addr(smem + s * G::kStage);
                const uint64_t dy = sdesc(base, 128, kCh), dx = sdesc(base + G::kY, 128, kCh);
                #pragma unroll
                for (int q = 0; q < 8; ++q)
                    mma_bf16(tmem, dy + uint64_t(q * 16), dx + uint64_t(q * 16), id,
                             it > 0 || q > 0 ? 1u : 0u);
                mma_commit(empty + s);
            }
            __syncwarp();
        }
        if (leader) {
            mma_commit(done);
            settle(done, 0);
        }
        __syncwarp();
    } else if (t0 < t1) {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        float *tile = reinterpret_cast<float *>(smem + G::kTile) + (warp - 2) * (32 * 17);
        if (warp_wait(done, 0, abort_flag, err)) {
            fence_after();
            float *dst = a.part + int64_t(blockIdx.z) * a.N * a.K;
            const uint32_t tq = tmem + (uint32_t(32 * quarter) << 16);
            #pragma unroll 1
            for (int c = 16 * half; c < G::BK; c += 32) {
                if (k0 + c >= a.K) break;
                float v[16];
                tmem_ld16(tq + uint32_t(c), v);
                #pragma unroll
                for (int e = 0; e < 16; ++e) tile[lane * 17 + e] = v[e];
                __syncwarp();
                const int e = lane & 15, k = k0 + c + e;
                #pragma unroll 4
                for (int q = lane >> 4; q < 32; q += 2) {
                    const int n = n0 + 32 * quarter + q;
                    if (n < a.N && k < a.K) dst[int64_t(n) * a.K + k] = tile[q * 17 + e];
                }
                __syncwarp();
            }
            fence_before();
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
}

struct FcPackArgs {
    FcPack seg[kMaxFcPack];
    int n;
};
__global__ void __launch_bounds__(256) fc_pack_kernel(const FcPackArgs a) {
    pdl_wait();
    const int64_t nth = int64_t(gridDim.x) * 256, tid = int64_t(blockIdx.x) * 256 + threadIdx.x;
    for (int s = 0; s < a.n; ++s) {
        const FcPack g = a.seg[s];
        const int kc = (g.K + 15) / 16 * 2;
        const uint32_t total = uint32_t((g.rows + g.BN - 1) / g.BN) * kc * g.BN;
        // one 16-byte unit (8 k of a row) per thread; neighbours take whichever
        // of rows and k is contiguous in W
        for (uint32_t u = uint32_t(tid); u < total; u += uint32_t(nth)) {
            uint32_t j, c, t;
            if (g.ks == 1) {
                c = u % kc;
                j = u / kc % g.BN;
                t = u / (uint32_t(kc) * g.BN);
            } else {
                j = u % g.BN;
                c = u / g.BN % kc;
                t = u / (uint32_t(kc) * g.BN);
            }
            const int row = int(t * g.BN + j);
            float v[8];
            #pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = int(c) * 8 + e;
                v[e] = row < g.rows && k < g.K ? __ldg(g.W + row * g.rs + k * g.ks) : 0.f;
            }
            *reinterpret_cast<uint4 *>(g.out + (int64_t(t * kc + c) * g.BN + j) * 16) =
                make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]),
                           pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
        }
    }
}

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// the offset layer: K = DIM, too short for the tensor cores; a thread computes
// 8 columns of a row, a warp stores 512 contiguous bytes
template <int DIM>
__global__ void __launch_bounds__(256) fc_offset_kernel(int64_t M, const float *__restrict__ off,
                                                        const float *__restrict__ W,
                                                        const float *__restrict__ b, FcMat r) {
    __shared__ float w[256 * DIM], bb[256];
    pdl_wait();
    for (int i = threadIdx.x; i < 256 * DIM; i += 256) w[i] = bf16r(__ldg(W + i));
    bb[threadIdx.x] = __ldg(b + threadIdx.x);
    __syncthreads();
    const int64_t units = (M + 127) / 128 * 128 * 32;
    for (int64_t u = int64_t(blockIdx.x) * 256 + threadIdx.x; u < units; u += int64_t(gridDim.x) * 256) {
        const int row = int(u & 127), c = int(u >> 7) & 31;
        const int64_t t = u >> 12, i = t * 128 + row;
        uint32_t h[4] = {0u, 0u, 0u, 0u};
        if (i < M) {
            float x[DIM], z[8];
            #pragma unroll
            for (int d = 0; d < DIM; ++d) x[d] = bf16r(__ldg(off + i * DIM + d));
            #pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int n = 8 * c + e;
                z[e] = 0.f;
                #pragma unroll
                for (int d = 0; d < DIM; ++d) z[e] = fmaf(x[d], w[n * DIM + d], z[e]);
                z[e] = fmaxf(z[e] + bb[n], 0.f);
            }
            #pragma unroll
            for (int e = 0; e < 4; ++e) h[e] = pack_bf16x2(z[2 * e], z[2 * e + 1]);
        }
        *reinterpret_cast<uint4 *>(r.p + t * r.tile + int64_t(r.chunk0 + c) * kCh + row * 16) =
            make_uint4(h[0], h[1], h[2], h[3]);
    }
}

// a block per row tile, a warp per chunk: lanes sum every 32nd row, then a
// butterfly over the lanes
template <int DIM>
__global__ void __launch_bounds__(256) fc_offset_grad_kernel(int64_t M,
                                                             const float *__restrict__ off,
                                                             FcMat gy, float *__restrict__ part) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = blockIdx.x;
    for (int c = threadIdx.x >> 5; c < 32; c += 8) {
        float s[8 * DIM];
        #pragma unroll
        for (int e = 0; e < 8 * DIM; ++e) s[e] = 0.f;
        for (int r = lane; r < 128; r += 32) {
            const int64_t i = t * 128 + r;
            if (i >= M) break;
            const uint4 g = __ldg(reinterpret_cast<const uint4 *>(
                gy.p + t * gy.tile + int64_t(gy.chunk0 + c) * kCh + r * 16));
            const uint32_t gw[4] = {g.x, g.y, g.z, g.w};
            #pragma unroll
            for (int d = 0; d < DIM; ++d) {
                const float x = bf16r(__ldg(off + i * DIM + d));
                #pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[(2 * e) * DIM + d] = fmaf(__uint_as_float(gw[e] << 16), x, s[(2 * e) * DIM + d]);
                    s[(2 * e + 1) * DIM + d] =
                        fmaf(__uint_as_float(gw[e] & 0xffff0000u), x, s[(2 * e + 1) * DIM + d]);
                }
            }
        }
        #pragma unroll
        for (int e = 0; e < 8 * DIM; ++e) {
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[e] += __shfl_xor_sync(kFull, s[e], o);
            if (lane == 0) part[t * 256 * DIM + c * 8 * DIM + e] = s[e];
        }
    }
}

// a few rows of a tiled matrix as row-major FP32 (fewer than an MMA's 16; larger
// products read the tiles)
__global__ void __launch_bounds__(256) fc_widen_kernel(FcMat A, int64_t M, float *__restrict__ out,
                                                       int64_t ld) {
    pdl_wait();
    const int64_t cols = int64_t(A.chunks) * 8;
    for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < M * cols; i += int64_t(gridDim.x) * 256) {
        const int64_t b = i / cols, c = i % cols;
        out[b * ld + c] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
            A.p + (b >> 7) * A.tile + (A.chunk0 + (c >> 3)) * kFcChunk + (b & 127) * 16 + (c & 7) * 2));
    }
}

template <int BN>
void launch_bn(const FcArgs &a, int sm_count, int *err, cudaStream_t st) {
    using G = FcGeo<BN>;
    cudaFuncSetAttribute(fc_gemm_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kTotal);
    launch_pdl(fc_gemm_kernel<BN>, dim3(std::min(a.mt * a.nt, sm_count)), dim3(kFcThreads),
               size_t(G::kTotal), st, a, err);
}

}  // namespace

// Columns of a tile: one tile for up to 96 (81 classes) and two for up to 352
// (343 classes: 176 each, 3% padding, where 256 + 87 would compute half as much
// again); otherwise the widest that still gives every SM a tile, as an MMA of 256
// columns takes 130 cycles and four of 64 take 200.
int fc_bn(int64_t M, int N, int sm_count) {
    if (N <= 96) return 96;
    if (N > 256 && N <= 352) return 176;
    const int64_t mt = (M + 127) / 128;
    if (mt * ((N + 255) / 256) >= sm_count) return 256;
    return mt * ((N + 127) / 128) >= sm_count * 3 / 4 ? 128 : 64;
}

void fc_split_like_gemm(int64_t M, int N, int K, int sm_count, int *nsplit, int *kc) {
    const int BN = N <= 32 ? 32 : N <= 128 ? 128 : N <= 144 ? 144 : N <= 256 ? 256 : 144;
    const int64_t tiles = (M + 127) / 128 * ((N + BN - 1) / BN), chunks = (K + 63) / 64;
    int64_t splits = 1;
    if (tiles < 2 * sm_count && chunks > 8)
        splits = std::min<int64_t>(chunks / 4, (2 * sm_count + tiles - 1) / tiles);
    *kc = int((chunks + splits - 1) / splits * 64);
    *nsplit = (K + *kc - 1) / *kc;
}

int launch_fc_pack(const FcPack *segs, int n, cudaStream_t st) {
    FcPackArgs a{};
    a.n = n;
    for (int i = 0; i < n; ++i) a.seg[i] = segs[i];
    launch_pdl(fc_pack_kernel, dim3(304), dim3(256), 0, st, a);
    return 1;
}

int launch_fc_gemm(const FcGemm &g, int *err, int sm_count, cudaStream_t st) {
    static_assert(kFcBiasMax % 16 == 0, "whole pieces of the bias");
    FcArgs a{};
    a.A = g.A;
    a.gate = g.gate;
    a.out = g.out;
    a.B = g.B;
    a.M = g.M;
    a.N = g.N;
    a.mt = int((g.M + 127) / 128);
    a.nt = (g.N + g.BN - 1) / g.BN;
    a.chunks = g.A.chunks;
    a.bias = g.bias;
    a.relu = g.relu ? 1 : 0;
    a.f32 = g.f32;
    a.ldf = g.ldf;
    a.colsum = g.colsum;
    a.nsplit = g.nsplit;
    a.split_stages = g.nsplit > 1 ? g.kc / 64 : 1;
    const int need = g.nsplit > 1 ? g.nsplit * g.BN : 2 * (g.BN <= 64 ? 64 : g.BN <= 128 ? 128 : 256);
    a.cols = need <= 128 ? 128 : need <= 256 ? 256 : 512;
    switch (g.BN) {
        case 64: launch_bn<64>(a, sm_count, err, st); break;
        case 96: launch_bn<96>(a, sm_count, err, st); break;
        case 128: launch_bn<128>(a, sm_count, err, st); break;
        case 176: launch_bn<176>(a, sm_count, err, st); break;
        default: launch_bn<256>(a, sm_count, err, st); break;
    }
    return 1;
}

int fc_wgrad_splits(int64_t M, int N, int K, int sm_count) {
    const int64_t rt = (M + 127) / 128;
    const int64_t tiles = int64_t((N + 127) / 128) * ((K + FcWgGeo::BK - 1) / FcWgGeo::BK);
    const int64_t most = std::max<int64_t>(1, sm_count / tiles);
    const int64_t per = (rt + std::min(rt, most) - 1) / std::min(rt, most);
    return int((rt + per - 1) / per);
}

int launch_fc_wgrad(const FcMat &Y, const FcMat &X, int64_t M, int N, int K, int splits,
                    float *part, int *err, cudaStream_t st) {
    FcWgArgs a{};
    a.Y = Y;
    a.X = X;
    a.row_tiles = (M + 127) / 128;
    a.N = N;
    a.K = K;
    a.per = int((a.row_tiles + splits - 1) / splits);
    a.part = part;
    cudaFuncSetAttribute(fc_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FcWgGeo::kTotal);
    launch_pdl(fc_wgrad_kernel,
               dim3((N + 127) / 128, (K + FcWgGeo::BK - 1) / FcWgGeo::BK, splits), dim3(kFcThreads),
               size_t(FcWgGeo::kTotal), st, a, err);
    return 1;
}

int launch_fc_widen(const FcMat &A, int64_t M, float *out, int64_t ld, cudaStream_t st) {
    const int64_t n = M * A.chunks * 8;
    launch_pdl(fc_widen_kernel, dim3(unsigned(std::min<int64_t>((n + 255) / 256, 64))), dim3(256), 0, st,
               A, M, out, ld);
    return 1;
}

int launch_fc_offset(int dim, int64_t M, const float *off, const float *W, const float *b,
                     const FcMat &r, int sm_count, cudaStream_t st) {
    const int64_t units = (M + 127) / 128 * 128 * 32;
    const int grid = int(std::min<int64_t>((units + 255) / 256, int64_t(sm_count) * 8));
    if (dim == 2)
        launch_pdl(fc_offset_kernel<2>, dim3(grid), dim3(256), 0, st, M, off, W, b, r);
    else
        launch_pdl(fc_offset_kernel<3>, dim3(grid), dim3(256), 0, st, M, off, W, b, r);
    return 1;
}

int launch_fc_offset_grad(int dim, int64_t M, const float *off, const FcMat &gy, float *part,
                          cudaStream_t st) {
    const int grid = int((M + 127) / 128);
    if (dim == 2)
        launch_pdl(fc_offset_grad_kernel<2>, dim3(grid), dim3(256), 0, st, M, off, gy, part);
    else
        launch_pdl(fc_offset_grad_kernel<3>, dim3(grid), dim3(256), 0, st, M, off, gy, part);
    return 1;
}

}  // namespace cs
