// Training of the convolutional networks on the tensor cores: every
// convolution's forward pass, weight gradient and input gradient as implicit
// GEMMs (tcgen05) without an im2col copy in global memory, and the
// regressor's head (both fully connected layers, the loss and their
// gradients) in one kernel.
//
// Tiles. A CTA takes G whole inputs whose G Po output positions fill the 128
// rows of an MMA tile (row = position of input 0, 1, ..). It keeps their
// activations in shared memory and lays the im2col operand A[row][k] out
// there, k = channel * taps + tap as the weights are stored. The operand
// layout [k / 8][row][k % 8] is K-major for the forward product (K = k) and,
// read with the transposed (MN-major) descriptor, the left operand of the first
// layer's weight gradient (K = row). The other layers' backward pass needs no
// im2col operand (conv_bwd_kernel below).
//
//   forward   z[row][o]  = sum_k A[row][k] W[o][k]        M = rows, N = 32
//   first     dW[k][o]   = sum_rows A[row][k] dz[row][o]  M = k,    N = 32
//
// The sums over k run in the K order and K = 16 steps of the general GEMM
// (tc_gemm.cu), those of the input gradient over the output channels and then
// the taps, in increasing order, so activations and input gradients are that
// path's bits. Weight gradients accumulate over a CTA's tiles in TMEM; the CTAs'
// partials are summed in a fixed order.
//
// What bounds the forward pass is not the tensor pipe but the operand build (a
// 16-byte shared load per tap and 8 channels, transposed in registers); global
// traffic is the BF16 activations and gradients alone. At a batch of 4096 the
// 2-D step's im2col, GEMM, col2im and ReLU kernels moved about 1.2 GB through
// FP32 buffers: a gradient call took 1102 us there and 1594 us for 2048 rows in
// 3-D, now 142 us and 212 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "tc_common.cuh"
#include "train_tc.h"

namespace cs {
namespace {

constexpr int kPitch = 40;        // halves per position in shared memory (5 x 16 bytes: no conflicts)
constexpr int kFwdThreads = 256;
constexpr int kWgThreads = 512;
constexpr int kRowsT = 128;       // MMA rows
constexpr int kChunk = kRowsT * 16;   // bytes of one 8-element K chunk of A

struct ConvArgs {
    const void *x;
    int64_t B, tiles;
    int G;                        // inputs per tile
    const uint8_t *w;             // packed weights of the pass
    // forward
    const float *bias;
    uint16_t *y;
    float *z;
    int nsplit, kc;               // K splits of the sum (kc a multiple of 64)
    // backward
    const uint16_t *dz;
    float *wpart, *bpart;
    uint16_t *dzp;
    int ring;                     // of y
};

// one layer's geometry: inputs of edge Si, channels first FP32 (First: the
// network's input, D channels) or [pos][32] BF16
template <int D, int SI, bool FIRST>
struct Geo {
    static constexpr int Dim = D, Si = SI, So = SI - 2;
    static constexpr bool First = FIRST;
    static constexpr int Pi = D == 2 ? Si * Si : Si * Si * Si;
    static constexpr int Po = D == 2 ? So * So : So * So * So;
    static constexpr int Taps = D == 2 ? 9 : 27;
    static constexpr int C = FIRST ? D : kTrainCh;
    static constexpr int K = C * Taps;
    static constexpr int Kp = (K + 15) / 16 * 16, Chunks = Kp / 8;
    static constexpr int GMax = kRowsT / Po;
    static constexpr int ActHalves = FIRST ? C * Pi : Pi * kPitch;   // per input
};

// shared memory of one CTA (bytes); the operand first
struct ConvSmem {
    int act, w, dz, tab, bar, total;
};

template <class N, bool BWD>
struct ConvCfg {
    static constexpr int D = N::Dim;
    // The operand is built in groups of 8 channels (Taps chunks of 8 columns;
    // the FP32 input's few columns all at once). A 2-D operand fits whole (four
    // groups); a 3-D one is built two groups at a time (an even number of
    // chunks: whole K = 16 steps).
    static constexpr int Groups = N::First ? 1 : 4;
    static constexpr int GroupChunks = N::First ? N::Chunks : N::Taps;
    static constexpr int Gb = N::First ? 1 : D == 2 ? 4 : 2;   // groups per build
    static constexpr int Cb = Gb * GroupChunks;
    static constexpr int Builds = Groups / Gb;
    static constexpr int Mt = (Cb + 15) / 16;                // weight-gradient M-tiles (first layer)
    static constexpr uint32_t Cols = 128;
    static constexpr int WBytes = !BWD ? N::Kp * kTrainCh * 2 : 0;
    // the classifier's layer, one input of 81 rows per tile, leaves room for a
    // second CTA per SM
    static constexpr int PerSm = BWD && N::Si == 11 ? 2 : 1;
    static_assert(!BWD || N::First, "weight gradient of the first layer alone");
    static_assert(BWD || Cb % 2 == 0, "whole K = 16 steps per build");
    static_assert(Builds * Gb == Groups && PerSm * Cols <= 512 && 32 * (BWD ? Mt : 1) <= int(Cols),
                  "whole builds, TMEM columns");
};

constexpr int kSmemMax = 232448, kSmemHalf = 113 * 1024;

template <class N, bool BWD>
constexpr ConvSmem conv_smem(int G) {
    using F = ConvCfg<N, BWD>;
    ConvSmem s{};
    s.act = F::Cb * kChunk;
    s.w = s.act + (G * N::ActHalves * 2 + 127) / 128 * 128;
    s.dz = s.w + F::WBytes;
    s.tab = s.dz + (BWD ? kTrainCh * kRowsT * 2 : 0);
    s.bar = (s.tab + (N::First ? N::Kp * 2 : 0) + 127) / 128 * 128;
    s.total = s.bar + 64;
    // an M-tile of the weight gradient reads 16 chunks from its first one,
    // past the built ones at the end (rows of no use): inside the allocation
    const int reach = F::Mt * 16 * kChunk;
    if (BWD && s.total < reach) s.total = reach;
    return s;
}

// The activations of inputs [b0, b0 + nb) on their way to shared memory:
// start() issues the loads, finish() makes them visible to the caller (the
// CTA still has to synchronise). BF16 activations travel as
// asynchronous copies into the padded rows; the network's FP32 input waits in
// registers and is rounded as it is stored, channels first.
template <class N, int NTH>
struct ActLoad {
    static constexpr int Regs = N::First ? (N::GMax * N::C * N::Pi + NTH - 1) / NTH : 1;
    float r[Regs];
    __device__ __forceinline__ void start(const ConvArgs &a, int64_t b0, int nb, uint8_t *act,
                                          int tid) {
        if constexpr (N::First) {
            const int n = nb * N::C * N::Pi;
            const float *src = static_cast<const float *>(a.x) + b0 * N::C * N::Pi;
            #pragma unroll
            for (int j = 0; j < Regs; ++j)
                r[j] = tid + j * NTH < n ? __ldg(src + tid + j * NTH) : 0.f;
        } else {
            const int n = nb * N::Pi * 4;
            const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(a.x) +
                                                               b0 * N::Pi * kTrainCh);
            for (int i = tid; i < n; i += NTH)
                cp_async16(act + (i >> 2) * (kPitch * 2) + (i & 3) * 16, src + i);
        }
    }
    __device__ __forceinline__ void finish(int nb, uint8_t *act, int tid) {
        if constexpr (N::First) {
            const int n = nb * N::C * N::Pi;
            #pragma unroll
            for (int j = 0; j < Regs; ++j)
                if (tid + j * NTH < n)
                    reinterpret_cast<__nv_bfloat16 *>(act)[tid + j * NTH] = __float2bfloat16_rn(r[j]);
        } else {
            cp_async_wait_all();
        }
    }
};

// offset (in halves) of operand column k of the network's input from its
// row's base, 0xffff past K
template <class N>
__device__ __forceinline__ void fill_tab(uint16_t *tab, int tid, int nth) {
    if constexpr (N::First)
        for (int k = tid; k < N::Kp; k += nth) {
            const int i = k / N::Taps, t = k % N::Taps;
            const int dx = t % 3, dy = (t / 3) % 3, dz = N::Dim == 3 ? t / 9 : 0;
            tab[k] = k >= N::K ? 0xffffu : uint16_t(i * N::Pi + (dz * N::Si + dy) * N::Si + dx);
        }
}

// base (in halves) of row r's window, -1 where the row holds no output
template <class N>
__device__ __forceinline__ int row_base(int nb, int r) {
    const int w = r / N::Po, p = r % N::Po;
    if (w >= nb) return -1;
    const int px = p % N::So, q = p / N::So;
    const int pb = N::Dim == 2 ? q * N::Si + px : ((q / N::So) * N::Si + q % N::So) * N::Si + px;
    return w * N::ActHalves + pb * (N::First ? 1 : kPitch);
}

// The im2col operand of the network's input into `dst`: a warp takes 32 rows
// of one chunk at a time, so its loads step by one position per lane.
template <class N, int NWARPS>
__device__ __forceinline__ void build_first(uint8_t *dst, const uint8_t *act, const uint16_t *tab,
                                            int base, int warp, int lane) {
    constexpr int Step = NWARPS / 4;
    const int row = 32 * (warp & 3) + lane;
    const uint16_t *s = reinterpret_cast<const uint16_t *>(act) + (base < 0 ? 0 : base);
    const uint32_t keep = base < 0 ? 0u : 0xffffffffu;
    #pragma unroll 3
    for (int i = 0; i < (N::Chunks + Step - 1) / Step; ++i) {
        const int c = (warp >> 2) + i * Step;
        if (c >= N::Chunks) break;
        const uint4 t = *reinterpret_cast<const uint4 *>(tab + 8 * c);
        const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
        uint32_t v[4];
        #pragma unroll
        for (int j = 0; j < 4; ++j) {   // zero past K
            const uint32_t k0 = tw[j] & 0xffffu, k1 = tw[j] >> 16;
            v[j] = (k0 == 0xffffu ? 0u : uint32_t(s[k0])) | (k1 == 0xffffu ? 0u : uint32_t(s[k1]) << 16);
        }
        *reinterpret_cast<uint4 *>(dst + c * kChunk + row * 16) =
            make_uint4(v[0] & keep, v[1] & keep, v[2] & keep, v[3] & keep);
    }
}

// tap t's offset in bytes from a row's base
template <class N>
__device__ __forceinline__ constexpr int tap_bytes(int t) {
    return (((N::Dim == 3 ? t / 9 : 0) * N::Si + (t / 3) % 3) * N::Si + t % 3) * kPitch * 2;
}

// halves i0 of a and i1 of b as one word
__device__ __forceinline__ uint32_t halves(uint32_t a, int i0, uint32_t b, int i1) {
    return __byte_perm(a, b, (i0 ? 0x32u : 0x10u) | ((i1 ? 0x76u : 0x54u) << 8));
}

// Part of a group of 8 channels of one row of the operand: column k = channel
// * Taps + tap of the group at chunk k / 8. 2-D: all of it; every tap's 8
// channels are one 16-byte load, transposed to (channel, tap) order in
// registers, and a chunk is one 16-byte store, conflict-free like the loads.
// 3-D: the group's channels 4 p .. 4 p + 3 (8-byte loads; 27 taps of 8 channels
// would not fit the registers), that is columns 108 p .. 108 p + 107: 13 chunks
// and half of the one in the middle. dst: the group's first chunk at the row;
// s: the row's window at the group's channels.
template <class N>
__device__ __forceinline__ void build_part(uint8_t *dst, const uint8_t *s, uint32_t keep, int p) {
    if constexpr (N::Dim == 2) {
        uint32_t v[9][4];
        #pragma unroll
        for (int t = 0; t < 9; ++t) {
            const uint4 q = *reinterpret_cast<const uint4 *>(s + tap_bytes<N>(t));
            v[t][0] = q.x & keep;
            v[t][1] = q.y & keep;
            v[t][2] = q.z & keep;
            v[t][3] = q.w & keep;
        }
        #pragma unroll
        for (int c = 0; c < 9; ++c) {
            uint32_t w[4];
            #pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k0 = 8 * c + 2 * j, k1 = k0 + 1;
                w[j] = halves(v[k0 % 9][k0 / 9 / 2], (k0 / 9) & 1, v[k1 % 9][k1 / 9 / 2], (k1 / 9) & 1);
            }
            *reinterpret_cast<uint4 *>(dst + c * kChunk) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        uint32_t v[27][2];
        #pragma unroll
        for (int t = 0; t < 27; ++t) {
            const uint2 q = *reinterpret_cast<const uint2 *>(s + tap_bytes<N>(t) + 8 * p);
            v[t][0] = q.x & keep;
            v[t][1] = q.y & keep;
        }
        auto word = [&](int k) {    // columns k, k + 1 of the part
            return halves(v[k % 27][k / 27 / 2], (k / 27) & 1, v[(k + 1) % 27][(k + 1) / 27 / 2],
                          ((k + 1) / 27) & 1);
        };
        if (p == 0) {
            #pragma unroll
            for (int c = 0; c < 13; ++c)
                *reinterpret_cast<uint4 *>(dst + c * kChunk) =
                    make_uint4(word(8 * c), word(8 * c + 2), word(8 * c + 4), word(8 * c + 6));
            *reinterpret_cast<uint2 *>(dst + 13 * kChunk) = make_uint2(word(104), word(106));
        } else {
            *reinterpret_cast<uint2 *>(dst + 13 * kChunk + 8) = make_uint2(word(0), word(2));
            #pragma unroll
            for (int c = 14; c < 27; ++c)
                *reinterpret_cast<uint4 *>(dst + c * kChunk) = make_uint4(
                    word(8 * c - 108), word(8 * c - 106), word(8 * c - 104), word(8 * c - 102));
        }
    }
}

// build j of the operand into `dst`
template <class N, bool BWD, int NWARPS>
__device__ __forceinline__ void build_operand(uint8_t *dst, const uint8_t *act, const uint16_t *tab,
                                              int base, int j, int warp, int lane) {
    using F = ConvCfg<N, BWD>;
    if constexpr (N::First) {
        build_first<N, NWARPS>(dst, act, tab, base, warp, lane);
    } else {
        const int row = 32 * (warp & 3) + lane;
        const uint8_t *s = act + (base < 0 ? 0 : base) * 2;
        constexpr int Parts = N::Dim == 2 ? 1 : 2;
        #pragma unroll 1
        for (int i = warp >> 2; i < F::Gb * Parts; i += NWARPS / 4) {
            const int g = i / Parts;
            build_part<N>(dst + g * F::GroupChunks * kChunk + row * 16, s + (j * F::Gb + g) * 16,
                          base < 0 ? 0u : 0xffffffffu, i % Parts);
        }
    }
}

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(slot)),
                 "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}

// wait (bounded) for the CTA's MMAs in flight, then release TMEM. Every
// thread of the CTA calls it; `bar` has no phase in use.
__device__ __forceinline__ void mma_drain(uint64_t *bar, uint32_t tmem, uint32_t cols, int warp) {
    if (warp == 0) {
        if (elect_one()) {
            mma_commit(bar);
            for (uint32_t i = 0; i < (1u << 24) && !mbar_try_wait(bar, 0); ++i)
                if (i > 64) __nanosleep(64);
        }
        __syncwarp();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_free(tmem, cols);
}

// a BF16 value above zero: an open ReLU
__device__ __forceinline__ bool positive(uint16_t h) { return h != 0 && h < 0x8000u; }

template <class N>
__global__ void __launch_bounds__(kFwdThreads, 2) conv_fwd_kernel(const ConvArgs a,
                                                                  const ConvSmem L, int *err) {
    using F = ConvCfg<N, false>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *act = smem + L.act, *wop = smem + L.w;
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem + L.tab);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.bar);   // MMAs, [2] the drain
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L.bar + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L.bar + 40);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t kCols = 128;
    constexpr int kNw = kFwdThreads / 32;

    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(bars + i, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(slot, kCols);
    fill_tab<N>(tab, tid, kFwdThreads);
    // the kernel before this one wrote its inputs
    pdl_wait();
    for (int i = tid; i < F::WBytes / 16; i += kFwdThreads) cp_async16(wop + 16 * i, a.w + 16 * i);
    ActLoad<N, kFwdThreads> ld;
    int64_t t = blockIdx.x;
    int nb = int(min(int64_t(a.G), a.B - t * a.G));
    ld.start(a, t * a.G, nb, act, tid);
    cp_async_wait_all();
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *slot;
    constexpr uint32_t id = idesc_bf16(128, 32);
    const uint64_t dw = sdesc(smem_addr(wop), kTrainCh * 16, 128);
    const int edge = N::So + 2 * a.ring;
    const int np = N::Dim == 2 ? edge * edge : edge * edge * edge;
    // this thread's output row and columns
    const int r = 32 * (warp & 3) + lane, o0 = 16 * (warp >> 2);
    const int ow = r / N::Po, op = r % N::Po;
    const int qx = op % N::So + a.ring, qy = (op / N::So) % N::So + a.ring;
    const int qz = N::Dim == 3 ? op / (N::So * N::So) + a.ring : 0;
    const int opos = (qz * edge + qy) * edge + qx;
    bool ok = true;
    int it = 0;
    while (t < a.tiles) {
        const int64_t b0 = t * a.G;
        ld.finish(nb, act, tid);
        const int base = row_base<N>(nb, r);
        fence_before();
        __syncthreads();
        fence_after();
        for (int j = 0; j < F::Builds && ok; ++j, ++it) {
            // the operand's previous MMAs are complete (with one build per tile
            // the tile before waited for them)
            if (F::Builds > 1 && it >= 1)
                ok = __syncthreads_and(mbar_wait(bars + 0, uint32_t(it - 1) & 1u, abort_flag, err));
            if (!ok) break;
            build_operand<N, false, kNw>(smem, act, tab, base, j, warp, lane);
            fence_async_smem();
            fence_before();
            __syncthreads();
            fence_after();
            if (warp == 0) {
                if (elect_one()) {
                    const uint64_t da = sdesc(smem_addr(smem), kChunk, 128);
                    const int c0 = j * F::Cb;
                    #pragma unroll
                    for (int q = 0; q < F::Cb / 2; ++q) {
                        const int k = 8 * c0 + 16 * q;
                        // at most three splits (kc >= K without any)
                        const int s = N::K > 512 ? (k >= a.kc) + (k >= 2 * a.kc) : 0;
                        mma_bf16(tmem + uint32_t(32 * s), da + uint64_t(2 * q * (kChunk >> 4)),
                                 dw + uint64_t((c0 + 2 * q) * kTrainCh), id,
                                 k - s * a.kc > 0 ? 1u : 0u);
                    }
                    mma_commit(bars + 0);
                }
                __syncwarp();
            }
        }
        if (!ok) break;
        // the activations are in the operand: fetch the next tile's
        const int nb_now = nb;
        t += gridDim.x;
        if (t < a.tiles) {
            nb = int(min(int64_t(a.G), a.B - t * a.G));
            ld.start(a, t * a.G, nb, act, tid);
        }
        // the tile's last build completes after all others
        ok = __syncthreads_and(mbar_wait(bars + 0, uint32_t(it - 1) & 1u, abort_flag, err));
        if (!ok) break;
        fence_after();
        const uint32_t tq = tmem + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(o0);
        float v[16];
        tmem_ld16(tq, v);
        if (N::K > 512 && a.nsplit > 1) {
            for (int s = 1; s < a.nsplit; ++s) {
                float u[16];
                tmem_ld16(tq + uint32_t(32 * s), u);
                #pragma unroll
                for (int e = 0; e < 16; ++e) v[e] += u[e];
            }
        }
        fence_before();
        if (ow < nb_now) {
            #pragma unroll
            for (int e = 0; e < 16; ++e) v[e] += __ldg(a.bias + o0 + e);
            if (a.y) {
                uint32_t h[8];
                #pragma unroll
                for (int e = 0; e < 8; ++e)
                    h[e] = pack_bf16x2(fmaxf(v[2 * e], 0.f), fmaxf(v[2 * e + 1], 0.f));
                uint4 *d = reinterpret_cast<uint4 *>(a.y + ((b0 + ow) * np + opos) * kTrainCh + o0);
                d[0] = make_uint4(h[0], h[1], h[2], h[3]);
                d[1] = make_uint4(h[4], h[5], h[6], h[7]);
            }
            if (a.z) {
                float4 *d = reinterpret_cast<float4 *>(a.z + ((b0 + ow) * N::Po + op) * kTrainCh + o0);
                #pragma unroll
                for (int e = 0; e < 4; ++e)
                    d[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            }
        }
    }
    cp_async_wait_all();
    mma_drain(bars + 2, tmem, kCols, warp);
}

// Weight gradient of the first layer (its input's gradient is not wanted): the
// im2col operand of a tile is built as in the forward pass and read with the
// transposed descriptor; the sum over all of a CTA's tiles stays in TMEM.
template <class N>
__global__ void __launch_bounds__(kWgThreads, ConvCfg<N, true>::PerSm) first_wgrad_kernel(
    const ConvArgs a, const ConvSmem L, int *err) {
    using F = ConvCfg<N, true>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *act = smem + L.act, *dzs = smem + L.dz;
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem + L.tab);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.bar);   // products, -, drain
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L.bar + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L.bar + 40);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(bars + i, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(slot, F::Cols);
    fill_tab<N>(tab, tid, kWgThreads);
    pdl_wait();
    ActLoad<N, kWgThreads> ld;
    int64_t t = blockIdx.x;
    int nb = int(min(int64_t(a.G), a.B - t * a.G));
    // dz of a tile: one 16-byte piece (8 channels of a row) per thread, the
    // next tile's fetched under this tile's products
    uint4 dzr;
    auto fetch_dz = [&]() {
        const int i = tid, rr = i >> 2;
        dzr = rr < nb * N::Po ? __ldg(reinterpret_cast<const uint4 *>(a.dz + t * a.G * N::Po * kTrainCh) + i)
                              : make_uint4(0u, 0u, 0u, 0u);
    };
    static_assert(kRowsT * 4 == kWgThreads, "one piece of dz per thread");
    ld.start(a, t * a.G, nb, act, tid);
    fetch_dz();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *slot;
    constexpr uint32_t id_w = idesc_mn(idesc_bf16(128, 32), true, true);
    const uint64_t dz_mn = sdesc(smem_addr(dzs), 128, kChunk);
    bool ok = true, any = false;
    uint32_t phase = 0;
    while (t < a.tiles) {
        ld.finish(nb, act, tid);
        *reinterpret_cast<uint4 *>(dzs + (tid & 3) * kChunk + (tid >> 2) * 16) = dzr;
        const int base = row_base<N>(nb, 32 * (warp & 3) + lane);
        __syncthreads();
        const int ksteps = (nb * N::Po + 15) / 16;
        t += gridDim.x;
        if (t < a.tiles) {
            nb = int(min(int64_t(a.G), a.B - t * a.G));
            fetch_dz();
        }
        build_first<N, kWgThreads / 32>(smem, act, tab, base, warp, lane);
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (warp == 0) {
            if (elect_one()) {
                #pragma unroll 1
                for (int mt = 0; mt < F::Mt; ++mt) {
                    const uint64_t da = sdesc(smem_addr(smem) + mt * 16 * kChunk, 128, kChunk);
                    #pragma unroll
                    for (int q = 0; q < kRowsT / 16; ++q)
                        if (q < ksteps)
                            mma_bf16(tmem + uint32_t(32 * mt), da + uint64_t(q * 16),
                                     dz_mn + uint64_t(q * 16), id_w, any || q > 0 ? 1u : 0u);
                }
                mma_commit(bars + 0);
            }
            __syncwarp();
        }
        // the input is not read again: fetch the next tile's
        if (t < a.tiles) ld.start(a, t * a.G, nb, act, tid);
        ok = __syncthreads_and(mbar_wait(bars + 0, phase, abort_flag, err));
        phase ^= 1u;
        fence_after();
        if (!ok) break;
        any = true;
    }
    if (ok && any && (warp >> 2) < 2) {
        // this CTA's weight gradient: rows of D are k, columns the output channel
        float *wp = a.wpart + int64_t(blockIdx.x) * N::K * kTrainCh;
        const int o0 = 16 * (warp >> 2);
        for (int mt = 0; mt < F::Mt; ++mt) {
            float v[16];
            tmem_ld16(tmem + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(32 * mt + o0), v);
            const int k = 128 * mt + 32 * (warp & 3) + lane;
            if (k < N::K) {
                #pragma unroll
                for (int e = 0; e < 16; ++e) wp[(o0 + e) * N::K + k] = v[e];
            }
        }
    }
    mma_drain(bars + 2, tmem, F::Cols, warp);
}

// ---------------------------------------------------------------------------
// Backward pass of the other layers, without an im2col operand. dz is laid out
// on the flat index of its input's positions, q = (z Si + y) Si + x of every
// input in turn, with zeros where no output position is: output position p of
// tap t then meets input position p + shift(t), shift = (dz Si + dy) Si + dx, and
// a tap is a row offset of an operand in shared memory.
//
//   columns  T_t[q][c] = sum_o dz[q - shift(t)][o] W[o][c][t]: M = 128 positions,
//            N = 32, K = 32, one product per tap into TMEM columns of its own.
//            dx[q][c] is the sum of the T_t in increasing t, each thread adding
//            its position's in registers: the same sums in the same order as
//            with the columns gradient in memory, with no gather (where the tap
//            leaves the output the product is 0: of finite weights).
//   weights  dW[(dy, o)][(dx, c)] += sum_q dz[q - Si dy][o] act[q + dx + Si^2 dz][c]:
//            M = 128 (3 x 32 used), N = 96, K = positions. Both operands are kept
//            in three copies, shifted by Si dy and by dx, so that the copies
//            continue the 8-channel chunks at one stride; 3-D adds dz by a row
//            offset, in TMEM columns of its own.
//
// Zero times a value that is not finite is no zero, so the products that no output
// position takes part in must not meet one. With weights that are not finite the
// epilogue adds only the taps that meet an output. An activation that is not finite
// is 1 in the operand, and the CTA adds its true products to its weight gradient
// at the end (add_nonfinite). Both are looked for as the operands are loaded; finite
// ones take the same path as before.
//
// Warps 0-7 add up T and mask it by the ReLU (warp w: positions 32 (w % 4) .. of
// the M-tile, 16 channels), warps 8-11 load, warp 12 issues the MMAs, handed over
// unit by unit by warp 13, which does its waiting. Two buffers of operands; the
// epilogue follows the tensor pipe three taps behind, and a slice of the weights'
// steps keeps the pipe busy until it has read a unit's last.
// Every wait is bounded (abort flag and device error flag).
//
// The tensor pipe needs 42 cycles for an MMA of N = 32 and 58 for N = 96, per tile
// of 250 positions 36 and 16 of them in 2-D (2.4k cycles), 54 and 24 per 125 in
// 3-D (3.7k). The kernel takes about twice that: a unit's products may not start
// before the unit before is read, and a commit is seen 250 cycles after the
// products, a part is read and added in 70. Measured: Si = 11 (4096 inputs) 36 us,
// Si = 7 20, 5 13.5, 3 9.8; 3-D (2048) Si = 5 56, Si = 3 23. With the im2col
// operand, dcol in shared memory and a gather from it: 108, 40, 18, 9.3; 72, 17.
// With the MMA warp waiting itself: 39, 21, 14, 9.6; 56, 23. T in two regions by
// turns, a hand-back per part, two M-tiles by turns, or one lane polling: 3-D
// Si = 5 63, 62, 74, 77.
// ---------------------------------------------------------------------------
constexpr int kBwdEpi = 8, kBwdLoad = 4, kBwdMma = kBwdEpi + kBwdLoad, kBwdSched = kBwdMma + 1;
constexpr int kBwdThreads = (kBwdSched + 1) * 32;

template <class N>
struct BwdCfg {
    static constexpr int D = N::Dim, Si = N::Si;
    static constexpr int RowsMax = D == 2 ? 256 : 128;        // positions of a tile
    static constexpr int GMax = RowsMax / N::Pi;
    // positions whose gradient leaves: the classifier's second layer has its
    // input's zero ring stored, which has none
    static constexpr int Ring = Si == 11 ? 1 : 0;
    static constexpr int Crop = Si - 2 * Ring;
    static constexpr int Np = D == 2 ? Crop * Crop : Crop * Crop * Crop;
    static constexpr int Planes = D == 2 ? 1 : 3;
    // T is computed a unit of taps at a time (the last one of 3-D shorter), and
    // UnitSteps steps of the weights' product follow each unit
    static constexpr int UnitTaps = D == 2 ? 9 : 7, Units = (N::Taps + UnitTaps - 1) / UnitTaps;
    static constexpr int Parts = (UnitTaps + 2) / 3, UnitSteps = 8 * Planes / Units;
    static_assert(UnitSteps * Units == 8 * Planes && UnitTaps % 3 <= 1, "whole slices, parts of three or one");
    static constexpr int Front = D == 2 ? 2 : 2 * Si * Si + 2;     // zero rows before dz
    // rows of a chunk: 2 mod 8, so that four chunks' stores meet no bank twice
    static constexpr int RowsA = (RowsMax + (D == 2 ? 0 : 2 * Si * Si) + 5) / 8 * 8 + 2;
    static constexpr int RowsZ = (Front + 2 * Si + RowsMax + 5) / 8 * 8 + 2;
    static constexpr int Kw = kTrainCh * N::Taps;             // rows of the weights
    static constexpr int ActB = 12 * RowsA * 16, DzB = 12 * RowsZ * 16;   // bytes of a buffer
    static constexpr int kAct = 2 * DzB;
    static constexpr int kW = kAct + 2 * ActB;
    static constexpr int kBar = kW + Kw * kTrainCh * 2;       // mbarriers: parts, 2 buffers, drain
    static constexpr int kCnt = kBar + (Parts + 3) * 8;       // u32 full [2], hdone [2], freed
    static constexpr uint32_t ColT = 96 * Planes;             // TMEM: weights, then a unit's T
    static constexpr int kSlot = kCnt + 5 * 4;                // TMEM address, abort flag, an
                                                              // activation that is not finite
    static constexpr int kRed = (kSlot + 12 + 15) / 16 * 16;  // f32 [8][16]
    static constexpr int kTotal = kRed + kBwdEpi * 16 * 4;
    static constexpr int PieceA = (GMax * N::Pi * 4 + kBwdLoad * 32 - 1) / (kBwdLoad * 32);
    static constexpr int PieceZ = (GMax * N::Po * 4 + kBwdLoad * 32 - 1) / (kBwdLoad * 32);
    static_assert(ColT + 32 * UnitTaps <= 512, "TMEM columns");
    static_assert(kTotal <= 232448, "shared memory of one CTA");
    // the last rows of M (a fourth copy of dz, never stored) are read from what
    // follows the buffer
    static_assert(DzB + 16 * RowsZ * 16 <= kTotal, "operand reads inside the allocation");
    static_assert(kTrainCh * (N::K + 1) * 4 <= kW, "the weight gradient's stage");
    static_assert(N::K * 3 * 4 <= kW, "add_nonfinite's masks");
};

// non-zero where a half of w is a BF16 infinity or NaN
__device__ __forceinline__ uint32_t nonfinite2(uint32_t w) {
    return ((w & 0x7fff7fffu) + 0x00800080u) & 0x80008000u;
}
__device__ __forceinline__ uint32_t nonfinite8(const uint4 v) {
    return nonfinite2(v.x) | nonfinite2(v.y) | nonfinite2(v.z) | nonfinite2(v.w);
}
// the halves of w that are not finite replaced by 1 of their sign
__device__ __forceinline__ uint32_t ones_for_nonfinite2(uint32_t w) {
    const uint32_t m = (nonfinite2(w) >> 15) * 0x7fffu;
    return (w & ~m) | (0x3f803f80u & m);
}

// The products of this CTA's activations that are not finite, into its weight
// gradient wp[o][K]: a warp takes an activation and a tap that meets an output,
// lane o its product with dz[o], an infinity or (with zero or NaN) a NaN. A sum of
// such terms and finite ones only depends on which of them occur, so each is one
// bit: mask [K][+Inf, -Inf, NaN], bit o. Runs only where the loader has met one.
template <class N>
__device__ __noinline__ void add_nonfinite(const uint16_t *act, const uint16_t *dz, int64_t B, int G,
                                           int n_mine, uint32_t *mask, float *wp) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < N::K * 3; i += kBwdThreads) mask[i] = 0;
    __syncthreads();
    for (int k = 0; k < n_mine; ++k) {
        const int64_t b0 = (blockIdx.x + int64_t(k) * gridDim.x) * G;
        const int n = int(min(int64_t(G), B - b0)) * N::Pi;
        const uint16_t *x = act + b0 * N::Pi * kTrainCh;
        for (int q = warp; q < n; q += kBwdThreads / 32) {
            const uint16_t mine = x[q * kTrainCh + lane];
            uint32_t bad = __ballot_sync(kFull, (mine & 0x7f80u) == 0x7f80u);
            const int w = q / N::Pi, p = q % N::Pi;
            const int px = p % N::Si, py = p / N::Si % N::Si, pz = N::Dim == 3 ? p / (N::Si * N::Si) : 0;
            for (; bad; bad &= bad - 1) {
                const int c = __ffs(bad) - 1;
                const float v = __uint_as_float(uint32_t(__shfl_sync(kFull, uint32_t(mine), c)) << 16);
                for (int t = 0; t < N::Taps; ++t) {
                    const int ox = px - t % 3, oy = py - t / 3 % 3, oz = N::Dim == 3 ? pz - t / 9 : 0;
                    if (unsigned(ox) >= unsigned(N::So) || unsigned(oy) >= unsigned(N::So) ||
                        unsigned(oz) >= unsigned(N::Dim == 3 ? N::So : 1))
                        continue;
                    uint32_t *m = mask + 3 * (c * N::Taps + t);
                    if (*static_cast<volatile uint32_t *>(m + 2) == 0xffffffffu) continue;
                    const int64_t r = (b0 + w) * N::Po + (oz * N::So + oy) * N::So + ox;
                    const float s = v * __uint_as_float(uint32_t(dz[r * kTrainCh + lane]) << 16);
                    const uint32_t pos = __ballot_sync(kFull, s > 0.f), neg = __ballot_sync(kFull, s < 0.f);
                    if (lane == 0) {
                        if (pos) atomicOr(m, pos);
                        if (neg) atomicOr(m + 1, neg);
                        if (~(pos | neg)) atomicOr(m + 2, ~(pos | neg));
                    }
                    __syncwarp();
                }
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < N::K * kTrainCh; i += kBwdThreads) {
        const uint32_t *m = mask + 3 * (i % N::K);
        const int o = i / N::K;
        const bool pos = (m[0] >> o) & 1u, neg = (m[1] >> o) & 1u, nan = (m[2] >> o) & 1u;
        const float inf = __int_as_float(0x7f800000);
        if (nan || (pos && neg))
            wp[i] += inf - inf;
        else if (pos || neg)
            wp[i] += pos ? inf : -inf;
    }
}

// Warp-uniform bounded wait for a phase that is a few hundred cycles away: polls
// without the suspension of try_wait (104 cycles a poll of a warp, 215 with it).
__device__ __forceinline__ bool spin_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          int *err) {
    const uint32_t addr = smem_addr(bar);
    for (uint32_t i = 0; i < (1u << 24); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (__all_sync(0xffffffffu, ok)) return true;
        if ((i & 255) == 255 && __any_sync(0xffffffffu, *abort_flag)) return false;
    }
    *abort_flag = 1;
    atomicExch(err, 1);
    return false;
}

// The scheduler warp hands a unit to the MMA warp on a named barrier; false for
// both where either's ok is. (A shared-memory load of the MMA warp itself returns
// only once its queued MMAs have drained.)
__device__ __forceinline__ bool handover(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.and.pred q, 1, 64, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"(uint32_t(ok))
        : "memory");
    return r != 0;
}

// whether any thread of the epilogue warps has the flag (named barrier 2)
__device__ __forceinline__ bool epi_or(bool flag) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, 2, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(r)
        : "r"(uint32_t(flag)), "n"(kBwdEpi * 32)
        : "memory");
    return r != 0;
}

// bounded wait for a phase that may be far away: sparse polls
__device__ __forceinline__ bool idle_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          int *err) {
    for (uint32_t i = 0; i < (1u << 22); ++i) {
        const bool ok = (threadIdx.x & 31) != 0 || mbar_try_wait(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (__any_sync(0xffffffffu, *abort_flag)) return false;
        __nanosleep(128);
    }
    *abort_flag = 1;
    atomicExch(err, 1);
    return false;
}

// 3 x 16 columns of FP32 from TMEM, 32 columns apart
__device__ __forceinline__ void tmem_ld16x3(uint32_t taddr, float (&v)[3][16]) {
    uint32_t r[48];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%48];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
        "%26, %27, %28, %29, %30, %31}, [%49];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, "
        "%42, %43, %44, %45, %46, %47}, [%50];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]),
          "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]),
          "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47])
        : "r"(taddr), "r"(taddr + 32u), "r"(taddr + 64u)
        : "memory");
    #pragma unroll
    for (int i = 0; i < 48; ++i) v[i / 16][i % 16] = __uint_as_float(r[i]);
}

template <class N>
__global__ void __launch_bounds__(kBwdThreads, 1) conv_bwd_kernel(const ConvArgs a, int *err) {
    using F = BwdCfg<N>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *dzs = smem, *acts = smem + F::kAct, *wop = smem + F::kW;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + F::kBar);
    uint64_t *done = bars + F::Parts, *drain = done + 2;
    // running counts (a warp is never a use ahead in one): loader warps that have
    // filled a buffer, epilogue warps that have read its activations, that have
    // read a unit's T
    uint32_t *full = reinterpret_cast<uint32_t *>(smem + F::kCnt);
    uint32_t *hdone = full + 2, *freed = full + 4;
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + F::kSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + F::kSlot + 4);
    volatile int *bad_act = abort_flag + 1;
    float *red = reinterpret_cast<float *>(smem + F::kRed);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < F::Parts + 3; ++i) mbar_init(bars + i, 1u);
        for (int i = 0; i < 5; ++i) full[i] = 0;
        *abort_flag = 0;
        *bad_act = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(slot, 512);
    for (int i = tid; i < F::kW / 16; i += kBwdThreads)
        reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    pdl_wait();
    for (int i = tid; i < F::Kw * kTrainCh * 2 / 16; i += kBwdThreads) cp_async16(wop + 16 * i, a.w + 16 * i);
    cp_async_wait_all();
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *slot;
    const int n_mine = int((a.tiles - 1 - blockIdx.x) / gridDim.x + 1);
    auto tile_b0 = [&](int k) { return (blockIdx.x + int64_t(k) * gridDim.x) * a.G; };
    auto tile_nb = [&](int k) { return int(min(int64_t(a.G), a.B - tile_b0(k))); };
    bool ok = true;

    if (warp == kBwdMma) {
        constexpr uint32_t id_c = idesc_bf16(128, 32);
        constexpr uint32_t id_w = idesc_mn(idesc_bf16(128, 96), true, true);
        const bool leader = elect_one();
        const uint64_t w_k = sdesc(smem_addr(wop), F::Kw * 16, 128);
        for (int k = 0; k < n_mine && ok; ++k) {
            const uint32_t zb = smem_addr(dzs + (k & 1) * F::DzB);
            // dz for T: the copy shifted by 2 Si; row q - shift is Front + 2 Si further on
            const uint64_t z_k = sdesc(zb + 8 * F::RowsZ * 16, F::RowsZ * 16, 128) + uint64_t(F::Front + 2 * N::Si);
            const uint64_t z_mn = sdesc(zb, 128, F::RowsZ * 16) + uint64_t(F::Front);
            const uint64_t a_mn = sdesc(smem_addr(acts + (k & 1) * F::ActB), 128, F::RowsA * 16);
            const int rows = tile_nb(k) * N::Pi, mts = (rows + 127) / 128, ksteps = (rows + 15) / 16;
            #pragma unroll 1
            for (int mt = 0; mt < mts && ok; ++mt) {
                #pragma unroll
                for (int u = 0; u < F::Units; ++u) {
                    ok = ok && handover(true);
                    fence_after();
                    if (ok && leader) {
                        // a value of its own, or the taps' descriptors are kept in
                        // registers over the tiles
                        uint64_t wt = w_k;
                        asm volatile("" : "+l"(wt));
                        #pragma unroll
                        for (int i = 0; i < F::UnitTaps && u * F::UnitTaps + i < N::Taps; ++i) {
                            const int t = u * F::UnitTaps + i;
                            const int sh = ((N::Dim == 3 ? t / 9 : 0) * N::Si + t / 3 % 3) * N::Si + t % 3;
                            #pragma unroll
                            for (int q = 0; q < 2; ++q)
                                mma_bf16(tmem + F::ColT + uint32_t(32 * i),
                                         z_k + uint64_t(128 * mt) + uint64_t(2 * q * F::RowsZ - sh),
                                         wt + uint64_t(32 * t + 2 * q * F::Kw), id_c, q > 0 ? 1u : 0u);
                            // the epilogue takes three taps at a time
                            if (i % 3 == 2 || i + 1 == F::UnitTaps) mma_commit(bars + i / 3);
                        }
                        #pragma unroll
                        for (int i = 0; i < F::UnitSteps; ++i) {
                            const int j = u * F::UnitSteps + i, pl = N::Dim == 2 ? 0 : j / 8;
                            const int q = N::Dim == 2 ? 8 * mt + j : j % 8;
                            if (q < ksteps)
                                mma_bf16(tmem + uint32_t(96 * pl), z_mn + uint64_t(16 * q),
                                         a_mn + uint64_t(16 * q + pl * N::Si * N::Si), id_w,
                                         (k | q) != 0 ? 1u : 0u);
                        }
                        if (u + 1 == F::Units && mt + 1 == mts) mma_commit(done + (k & 1));
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp == kBwdSched) {
        uint32_t n = 0;                                  // units so far
        for (int k = 0; k < n_mine && ok; ++k) {
            const int units = (tile_nb(k) * N::Pi + 127) / 128 * F::Units;
            for (int u = 0; u < units && ok; ++u, ++n) {
                // the operands are in place; the unit before is read
                ok = (u > 0 || wait_count(full + (k & 1), uint32_t(kBwdLoad * (k / 2 + 1)), abort_flag, err)) &&
                     wait_count(freed, kBwdEpi * n, abort_flag, err);
                ok = handover(ok);
            }
        }
    } else if (warp >= kBwdEpi) {
        const int lt = tid - kBwdEpi * 32;
        for (int k = 0; k < n_mine; ++k) {
            const int64_t b0 = tile_b0(k);
            const int nb = tile_nb(k);
            const uint4 *xa = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(a.x) + b0 * N::Pi * kTrainCh);
            const uint4 *xz = reinterpret_cast<const uint4 *>(a.dz + b0 * N::Po * kTrainCh);
            uint4 va[F::PieceA], vz[F::PieceZ];
            #pragma unroll
            for (int j = 0; j < F::PieceZ; ++j) {
                const int i = lt + j * kBwdLoad * 32;
                vz[j] = i < nb * N::Po * 4 ? __ldg(xz + i) : make_uint4(0u, 0u, 0u, 0u);
            }
            #pragma unroll
            for (int j = 0; j < F::PieceA; ++j) {
                const int i = lt + j * kBwdLoad * 32;
                va[j] = i < nb * N::Pi * 4 ? __ldg(xa + i) : make_uint4(0u, 0u, 0u, 0u);
            }
            // the tile before last is done with this buffer
            if (k >= 2)
                ok = idle_wait(done + (k & 1), uint32_t(k / 2 - 1) & 1u, abort_flag, err) &&
                     wait_count(hdone + (k & 1), uint32_t(kBwdEpi * (k / 2)), abort_flag, err);
            if (!ok) break;
            uint8_t *zb = dzs + (k & 1) * F::DzB, *ab = acts + (k & 1) * F::ActB;
            #pragma unroll
            for (int j = 0; j < F::PieceZ; ++j) {
                const int i = lt + j * kBwdLoad * 32;
                if (i >= a.G * N::Po * 4) break;          // inputs past the batch: zeros
                const int p = i >> 2, w = p / N::Po, o = p % N::Po;
                const int q = w * N::Pi + (N::Dim == 2 ? o / N::So * N::Si + o % N::So
                                                       : (o / (N::So * N::So) * N::Si + o / N::So % N::So) * N::Si + o % N::So);
                #pragma unroll
                for (int c = 0; c < 3; ++c)
                    *reinterpret_cast<uint4 *>(zb + ((4 * c + (i & 3)) * F::RowsZ + F::Front + q + c * N::Si) * 16) = vz[j];
            }
            auto put_act = [&](int j, const uint4 v) {
                const int i = lt + j * kBwdLoad * 32, q = i >> 2;
                if (i >= a.G * N::Pi * 4) return;
                #pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (q >= c) *reinterpret_cast<uint4 *>(ab + ((4 * c + (i & 3)) * F::RowsA + q - c) * 16) = v;
            };
            uint32_t top = 0;     // the largest half: activations come from a ReLU, none is negative
            #pragma unroll
            for (int j = 0; j < F::PieceA; ++j) {
                put_act(j, va[j]);
                top = __vmaxu2(top, __vmaxu2(__vmaxu2(va[j].x, va[j].y), __vmaxu2(va[j].z, va[j].w)));
            }
            if (nonfinite2(top)) {
                *bad_act = 1;
                #pragma unroll
                for (int j = 0; j < F::PieceA; ++j)
                    put_act(j, make_uint4(ones_for_nonfinite2(va[j].x), ones_for_nonfinite2(va[j].y),
                                          ones_for_nonfinite2(va[j].z), ones_for_nonfinite2(va[j].w)));
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) red_release_add(full + (k & 1), 1u);
        }
    } else {
        const int wq = warp & 3, ch = 2 * (warp >> 2);   // lane quarter, first 8-channel chunk
        const uint32_t tq = tmem + F::ColT + (uint32_t(32 * wq) << 16) + uint32_t(8 * ch);
        float db[16];
        #pragma unroll
        for (int e = 0; e < 16; ++e) db[e] = 0.f;
        uint32_t ph = 0;                                 // phases of the parts' barriers
        // weights that are not finite, while the first tile is on its way
        uint32_t bad = 0;
        for (int i = tid; i < F::Kw * kTrainCh * 2 / 16; i += kBwdEpi * 32)
            bad |= nonfinite8(reinterpret_cast<const uint4 *>(wop)[i]);
        const bool bad_w = epi_or(bad != 0);
        for (int k = 0; k < n_mine && ok; ++k) {
            const int64_t b0 = tile_b0(k);
            const int rows = tile_nb(k) * N::Pi, mts = (rows + 127) / 128;
            const uint8_t *h = acts + (k & 1) * F::ActB + ch * F::RowsA * 16;
            for (int mt = 0; mt < mts && ok; ++mt) {
                float s[16];
                #pragma unroll
                for (int e = 0; e < 16; ++e) s[e] = 0.f;
                // the sum of a position's T_t; masked: of the taps that meet an output
                auto sum_taps = [&](auto m) {
                    constexpr bool masked = decltype(m)::value;
                    uint32_t meets = 0xffffffffu;        // bit t: tap t
                    if (masked) {
                        const int o = (128 * mt + 32 * wq + lane) % N::Pi;
                        const int x = o % N::Si, y = o / N::Si % N::Si, z = o / (N::Si * N::Si);
                        #pragma unroll
                        for (int t = 0; t < N::Taps; ++t)
                            if (unsigned(x - t % 3) >= unsigned(N::So) || unsigned(y - t / 3 % 3) >= unsigned(N::So) ||
                                (N::Dim == 3 && unsigned(z - t / 9) >= unsigned(N::So)))
                                meets &= ~(1u << t);
                    }
                    #pragma unroll 1
                    for (int u = 0; u < F::Units && ok; ++u) {
                        const int taps = min(F::UnitTaps, N::Taps - u * F::UnitTaps);
                        #pragma unroll
                        for (int g = 0; g < F::Parts; ++g) {
                            // (the last unit may have a part less)
                            if (3 * g >= taps) break;
                            ok = spin_wait(bars + g, (ph >> g) & 1u, abort_flag, err);
                            if (!ok) break;
                            ph ^= 1u << g;
                            fence_after();
                            const uint32_t part = meets >> (u * F::UnitTaps + 3 * g);
                            if (F::UnitTaps - 3 * g >= 3) {
                                float v[3][16];
                                tmem_ld16x3(tq + uint32_t(96 * g), v);
                                #pragma unroll
                                for (int i = 0; i < 3; ++i)
                                    #pragma unroll
                                    for (int e = 0; e < 16; ++e)
                                        s[e] += !masked || ((part >> i) & 1u) ? v[i][e] : 0.f;
                            } else {
                                float v[16];
                                tmem_ld16(tq + uint32_t(96 * g), v);
                                #pragma unroll
                                for (int e = 0; e < 16; ++e) s[e] += !masked || (part & 1u) ? v[e] : 0.f;
                            }
                        }
                        fence_before();
                        __syncwarp();
                        if (lane == 0) red_release_add(freed, 1u);
                    }
                };
                if (bad_w)
                    sum_taps(std::true_type());
                else
                    sum_taps(std::false_type());
                if (!ok) break;
                const int p = 128 * mt + 32 * wq + lane, w = p / N::Pi, o = p % N::Pi;
                const int x = o % N::Si - F::Ring, y = (o / N::Si) % N::Si - F::Ring;
                bool in = p < rows;
                int64_t op = b0 * N::Pi + p;
                if (F::Ring) {
                    in = in && unsigned(x) < unsigned(F::Crop) && unsigned(y) < unsigned(F::Crop);
                    op = (b0 + w) * F::Np + y * F::Crop + x;
                }
                // the activations are in place (the loaders' stores, seen through `full`)
                if (mt == 0) ok = wait_count(full + (k & 1), uint32_t(kBwdLoad * (k / 2 + 1)), abort_flag, err);
                if (!ok) break;
                if (in) {
                    uint4 *out = reinterpret_cast<uint4 *>(a.dzp + op * kTrainCh + 8 * ch);
                    #pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const uint4 hq = *reinterpret_cast<const uint4 *>(h + (c * F::RowsA + p) * 16);
                        const uint32_t hw[4] = {hq.x, hq.y, hq.z, hq.w};
                        uint32_t r[4];
                        #pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            // through the ReLU of the layer below: its output is positive
                            const float v0 = positive(uint16_t(hw[e])) ? s[8 * c + 2 * e] : 0.f;
                            const float v1 = positive(uint16_t(hw[e] >> 16)) ? s[8 * c + 2 * e + 1] : 0.f;
                            db[8 * c + 2 * e] += v0;
                            db[8 * c + 2 * e + 1] += v1;
                            r[e] = pack_bf16x2(v0, v1);
                        }
                        out[c] = make_uint4(r[0], r[1], r[2], r[3]);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) red_release_add(hdone + (k & 1), 1u);
        }
        // column sums of the input gradient: a warp's lanes, then the warps in order
        #pragma unroll
        for (int e = 0; e < 16; ++e) {
            #pragma unroll
            for (int m = 16; m > 0; m >>= 1) db[e] += __shfl_xor_sync(0xffffffffu, db[e], m);
            if (lane == 0) red[warp * 16 + e] = db[e];
        }
    }
    // wait (bounded) for the MMAs in flight; the weight gradient is complete
    if (warp == kBwdMma) {
        if (elect_one()) {
            mma_commit(drain);
            for (uint32_t i = 0; i < (1u << 24) && !mbar_try_wait(drain, 0); ++i)
                if (i > 64) __nanosleep(64);
        }
        __syncwarp();
    }
    fence_before();
    const bool good = __syncthreads_and(ok && !*abort_flag) != 0;
    fence_after();
    if (good) {
        // this CTA's weight gradient through shared memory in the weights' layout:
        // D's lanes are (line dy, output channel), columns (dx, input channel)
        float *stage = reinterpret_cast<float *>(smem);
        const int dy = warp & 3;
        if (warp < kBwdEpi && dy < 3) {
            const int c0 = 16 * (warp >> 2);
            #pragma unroll 1
            for (int pl = 0; pl < F::Planes; ++pl) {
                float v[3][16];
                tmem_ld16x3(tmem + (uint32_t(32 * dy) << 16) + uint32_t(96 * pl + c0), v);
                float *st = stage + lane * (N::K + 1) + (3 * pl + dy) * 3;
                #pragma unroll
                for (int e = 0; e < 16; ++e)
                    #pragma unroll
                    for (int dx = 0; dx < 3; ++dx) st[(c0 + e) * N::Taps + dx] = v[dx][e];
            }
        }
        __syncthreads();
        float *wp = a.wpart + int64_t(blockIdx.x) * N::K * kTrainCh;
        for (int i = tid; i < N::K * kTrainCh; i += kBwdThreads) wp[i] = stage[i / N::K * (N::K + 1) + i % N::K];
        if (tid < kTrainCh) {
            const float *r = red + (tid / 16) * 64 + tid % 16;
            a.bpart[int64_t(blockIdx.x) * kTrainCh + tid] = ((r[0] + r[16]) + r[32]) + r[48];
        }
        if (*bad_act) {
            __syncthreads();                             // the stage is read
            add_nonfinite<N>(static_cast<const uint16_t *>(a.x), a.dz, a.B, a.G, n_mine,
                             reinterpret_cast<uint32_t *>(smem), wp);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_free(tmem, 512);
}

// Weights of one convolution (FP32 W[32][K]) as the operands of both passes:
// forward bf16 [Kp / 8][32][8] (zero past K) and, with dgrad, backward [4][Kw][8],
// row 32 tap + channel.
// Weights of fc1 (W1[256][32]) the same way: bf16 [4][256][8].
struct PackArgs {
    PackSeg seg[kMaxPack];
    int n;
};
__global__ void __launch_bounds__(256) pack_train_kernel(const PackArgs a) {
    const int nth = gridDim.x * 256, tid = blockIdx.x * 256 + threadIdx.x;
    pdl_wait();
    for (int s = 0; s < a.n; ++s) {
        const PackSeg &g = a.seg[s];
        const int kp = (g.K + 15) / 16 * 16;
        __nv_bfloat16 *f = reinterpret_cast<__nv_bfloat16 *>(g.fwd);
        if (f)
            for (int e = tid; e < kTrainCh * kp; e += nth) {
                const int j = e & 7, o = (e >> 3) & 31, k = (e >> 8) * 8 + j;
                f[e] = __float2bfloat16_rn(k < g.K ? __ldg(g.W + o * g.K + k) : 0.f);
            }
        __nv_bfloat16 *b = reinterpret_cast<__nv_bfloat16 *>(g.bwd);
        if (b)
            for (int e = tid; e < kTrainCh * g.kw; e += nth) {
                const int j = e & 7, k = (e >> 3) % g.kw, o = (e >> 3) / g.kw * 8 + j;
                // row k: tap k / 32, channel k % 32
                b[e] = __float2bfloat16_rn(__ldg(g.W + o * g.K + k % kTrainCh * (g.K / kTrainCh) + k / kTrainCh));
            }
        __nv_bfloat16 *h = reinterpret_cast<__nv_bfloat16 *>(g.fc1);
        if (h)
            for (int e = tid; e < kTrainCh * 256; e += nth) {
                const int j = e & 7, n = (e >> 3) & 255, c = (e >> 11) * 8 + j;
                h[e] = __float2bfloat16_rn(__ldg(g.W + n * kTrainCh + c));
            }
    }
}

// ---------------------------------------------------------------------------
// The regressor's head. A CTA takes R (32, 64 or 128) rows; an MMA tile has
// 128, but the row count only bounds the K = row products, and small tiles
// spread a batch over more SMs (the two serial passes over the 256 hidden
// units are what a CTA spends its time on).
// ---------------------------------------------------------------------------
constexpr int kHid = 256;

struct HeadSmem {
    static constexpr int kH = 0;                               // h: bf16 [4][128][8]
    static constexpr int kW1 = kH + 4 * kChunk;                // W1: bf16 [4][256][8]
    static constexpr int kA5 = kW1 + 4 * kHid * 16;            // a5: bf16 [32][128][8]
    static constexpr int kDa = kA5 + 32 * kChunk;              // da5: the same
    static constexpr int kGop = kDa + 32 * kChunk;             // gout: bf16 [2][128][8]
    static constexpr int kG = kGop + 2 * kChunk;               // gout rounded to BF16: f32 [128][4]
    static constexpr int kGf = kG + kRowsT * 16;               // gout: f32 [128][4]
    static constexpr int kW2 = kGf + kRowsT * 16;              // W2 rounded to BF16: f32 [3][256]
    static constexpr int kB1 = kW2 + 3 * kHid * 4;             // f32 [256]
    static constexpr int kRed = kB1 + kHid * 4;                // f32 [128]
    static constexpr int kBar = kRed + kRowsT * 4;
    static constexpr int kTotal = kBar + 64;
};
static_assert(HeadSmem::kTotal <= 232448, "shared memory of one CTA");

struct HeadArgs {
    int64_t B;
    int R;
    const uint16_t *h;
    const uint8_t *w1;            // packed W1
    const float *b1, *W2, *b2, *tgt;
    float *out;
    uint16_t *dz;
    float *part;
};

template <int DIM>
__global__ void __launch_bounds__(256, 1) head_train_kernel(const HeadArgs a, int *err) {
    using S = HeadSmem;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + S::kBar);
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + S::kBar + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + S::kBar + 40);
    float *g = reinterpret_cast<float *>(smem + S::kG), *gf = reinterpret_cast<float *>(smem + S::kGf);
    float *w2 = reinterpret_cast<float *>(smem + S::kW2);
    float *b1 = reinterpret_cast<float *>(smem + S::kB1);
    float *red = reinterpret_cast<float *>(smem + S::kRed);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t kCols = 512, kDy = 256, kDw1 = 288, kDw2 = 352;
    const int64_t r0 = int64_t(blockIdx.x) * a.R;
    const int rows = int(min(int64_t(a.R), a.B - r0));
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(bars + i, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(slot, kCols);
    pdl_wait();
    for (int i = tid; i < kRowsT * 4; i += 256) {
        const int r = i >> 2, q = i & 3;
        const uint4 *src = reinterpret_cast<const uint4 *>(a.h + r0 * kTrainCh);
        *reinterpret_cast<uint4 *>(smem + S::kH + q * kChunk + r * 16) =
            r < rows ? __ldg(src + i) : make_uint4(0u, 0u, 0u, 0u);
    }
    for (int i = tid; i < kHid * kTrainCh / 8; i += 256)
        cp_async16(smem + S::kW1 + 16 * i, a.w1 + 16 * i);
    for (int i = tid; i < 2 * kChunk / 16; i += 256)
        reinterpret_cast<uint4 *>(smem + S::kGop)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < DIM * kHid; i += 256)
        w2[i] = __bfloat162float(__float2bfloat16_rn(__ldg(a.W2 + i)));
    b1[tid] = __ldg(a.b1 + tid);
    cp_async_wait_all();
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *slot;
    const uint64_t h_k = sdesc(smem_addr(smem + S::kH), kChunk, 128);
    const uint64_t h_mn = sdesc(smem_addr(smem + S::kH), 128, kChunk);
    const uint64_t w1_k = sdesc(smem_addr(smem + S::kW1), kHid * 16, 128);
    const uint64_t w1_mn = sdesc(smem_addr(smem + S::kW1), 128, kHid * 16);
    if (warp == 0) {
        if (elect_one()) {
            for (int q = 0; q < 2; ++q)
                mma_bf16(tmem, h_k + uint64_t(2 * q * (kChunk >> 4)), w1_k + uint64_t(2 * q * kHid),
                         idesc_bf16(128, 256), q > 0 ? 1u : 0u);
            mma_commit(bars + 0);
        }
        __syncwarp();
    }
    bool ok = __syncthreads_and(mbar_wait(bars + 0, 0u, abort_flag, err));
    if (ok) {
        fence_after();
        // ---- a thread per row: a5 = ReLU(z5), the output, its gradient ----
        float sq = 0.f;
        if (warp < 4 && 32 * warp < a.R) {
            const int r = tid;
            float acc[DIM];
            #pragma unroll
            for (int d = 0; d < DIM; ++d) acc[d] = 0.f;
            #pragma unroll 1
            for (int n0 = 0; n0 < kHid; n0 += 16) {
                float v[16];
                tmem_ld16(tmem + (uint32_t(32 * warp) << 16) + uint32_t(n0), v);
                uint32_t hv[8];
                #pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 bb = *reinterpret_cast<const float4 *>(b1 + n0 + 4 * q);
                    const float z[4] = {v[4 * q] + bb.x, v[4 * q + 1] + bb.y, v[4 * q + 2] + bb.z,
                                        v[4 * q + 3] + bb.w};
                    hv[2 * q] = pack_bf16x2(fmaxf(z[0], 0.f), fmaxf(z[1], 0.f));
                    hv[2 * q + 1] = pack_bf16x2(fmaxf(z[2], 0.f), fmaxf(z[3], 0.f));
                    const float hf[4] = {__uint_as_float(hv[2 * q] << 16),
                                         __uint_as_float(hv[2 * q] & 0xffff0000u),
                                         __uint_as_float(hv[2 * q + 1] << 16),
                                         __uint_as_float(hv[2 * q + 1] & 0xffff0000u)};
                    #pragma unroll
                    for (int d = 0; d < DIM; ++d) {
                        const float4 ww = *reinterpret_cast<const float4 *>(w2 + d * kHid + n0 + 4 * q);
                        acc[d] = fmaf(hf[0], ww.x, acc[d]);
                        acc[d] = fmaf(hf[1], ww.y, acc[d]);
                        acc[d] = fmaf(hf[2], ww.z, acc[d]);
                        acc[d] = fmaf(hf[3], ww.w, acc[d]);
                    }
                }
                if (a.tgt) {
                    // rows past the batch are zero: they meet zeros, and
                    // ReLU(b1) need not be finite
                    const uint32_t keep = r < rows ? 0xffffffffu : 0u;
                    uint8_t *d = smem + S::kA5 + (n0 >> 3) * kChunk + r * 16;
                    *reinterpret_cast<uint4 *>(d) =
                        make_uint4(hv[0] & keep, hv[1] & keep, hv[2] & keep, hv[3] & keep);
                    *reinterpret_cast<uint4 *>(d + kChunk) =
                        make_uint4(hv[4] & keep, hv[5] & keep, hv[6] & keep, hv[7] & keep);
                }
            }
            fence_before();
            #pragma unroll
            for (int d = 0; d < DIM; ++d) {
                const float o = acc[d] + __ldg(a.b2 + d);
                float gd = 0.f;
                if (r < rows) {
                    a.out[(r0 + r) * DIM + d] = o;
                    if (a.tgt) {
                        const float e = o - __ldg(a.tgt + (r0 + r) * DIM + d);
                        gd = 2.f * e / float(a.B * DIM);
                        sq += e * e;
                    }
                }
                if (a.tgt) {
                    const __nv_bfloat16 gb = __float2bfloat16_rn(gd);
                    gf[r * 4 + d] = gd;
                    g[r * 4 + d] = __bfloat162float(gb);
                    reinterpret_cast<__nv_bfloat16 *>(smem + S::kGop)[r * 8 + d] = gb;
                }
            }
            red[r] = sq;
        }
    }
    if (ok && a.tgt) {
        float *part = a.part + int64_t(blockIdx.x) * (kHid * kTrainCh + kHid + DIM * kHid + DIM +
                                                      kTrainCh + 1);
        float *p_b1 = part + kHid * kTrainCh, *p_w2 = p_b1 + kHid, *p_b2 = p_w2 + DIM * kHid;
        float *p_db = p_b2 + DIM, *p_loss = p_db + kTrainCh;
        __syncthreads();
        // ---- a thread per hidden unit: da5 = W2^T gout through the ReLU ----
        {
            float w[DIM], s = 0.f;
            #pragma unroll
            for (int d = 0; d < DIM; ++d) w[d] = w2[d * kHid + tid];
            const uint16_t *a5 = reinterpret_cast<const uint16_t *>(smem + S::kA5) +
                                 (tid >> 3) * (kChunk / 2) + (tid & 7);
            __nv_bfloat16 *da = reinterpret_cast<__nv_bfloat16 *>(smem + S::kDa) +
                                (tid >> 3) * (kChunk / 2) + (tid & 7);
            #pragma unroll 4
            for (int r = 0; r < a.R; ++r) {
                float v = 0.f;
                #pragma unroll
                for (int d = 0; d < DIM; ++d) v = fmaf(g[r * 4 + d], w[d], v);
                v = positive(a5[r * 8]) ? v : 0.f;
                s += v;
                da[r * 8] = __float2bfloat16_rn(v);
            }
            p_b1[tid] = s;
            if (tid < DIM) {
                float t = 0.f;
                for (int r = 0; r < a.R; ++r) t += gf[r * 4 + tid];
                p_b2[tid] = t;
            }
            if (tid == 32) {
                float t = 0.f;
                for (int r = 0; r < a.R; ++r) t += red[r];
                *p_loss = t;
            }
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (warp == 0) {
            if (elect_one()) {
                const uint64_t da_k = sdesc(smem_addr(smem + S::kDa), kChunk, 128);
                // dy[row][c] = sum_n da5[row][n] W1[n][c]
                for (int q = 0; q < kHid / 16; ++q)
                    mma_bf16(tmem + kDy, da_k + uint64_t(2 * q * (kChunk >> 4)),
                             w1_mn + uint64_t(q * 16), idesc_mn(idesc_bf16(128, 32), false, true),
                             q > 0 ? 1u : 0u);
                for (int mt = 0; mt < 2; ++mt) {
                    const uint64_t da_mn =
                        sdesc(smem_addr(smem + S::kDa) + mt * 16 * kChunk, 128, kChunk);
                    const uint64_t a5_mn =
                        sdesc(smem_addr(smem + S::kA5) + mt * 16 * kChunk, 128, kChunk);
                    const uint64_t g_mn = sdesc(smem_addr(smem + S::kGop), 128, kChunk);
                    for (int q = 0; q < a.R / 16; ++q) {
                        // dW1[n][c] = sum_rows da5[row][n] h[row][c]
                        mma_bf16(tmem + kDw1 + uint32_t(32 * mt), da_mn + uint64_t(q * 16),
                                 h_mn + uint64_t(q * 16), idesc_mn(idesc_bf16(128, 32), true, true),
                                 q > 0 ? 1u : 0u);
                        // dW2[d][n] = sum_rows gout[row][d] a5[row][n]
                        mma_bf16(tmem + kDw2 + uint32_t(16 * mt), a5_mn + uint64_t(q * 16),
                                 g_mn + uint64_t(q * 16), idesc_mn(idesc_bf16(128, 16), true, true),
                                 q > 0 ? 1u : 0u);
                    }
                }
                mma_commit(bars + 1);
            }
            __syncwarp();
        }
        ok = __syncthreads_and(mbar_wait(bars + 1, 0u, abort_flag, err));
        if (ok) {
            fence_after();
            const uint32_t tq = tmem + (uint32_t(32 * (warp & 3)) << 16);
            float *st = reinterpret_cast<float *>(smem + S::kA5);   // [128][33], MMAs complete
            if (warp < 4) {
                float v[32];
                tmem_ld32(tq + kDy, v);
                const int r = tid;
                uint32_t hv[16];
                #pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const uint16_t hb = reinterpret_cast<const uint16_t *>(
                        smem + S::kH + (c >> 3) * kChunk + r * 16)[c & 7];
                    v[c] = positive(hb) && r < rows ? v[c] : 0.f;
                    st[r * 33 + c] = v[c];
                }
                if (r < rows) {
                    #pragma unroll
                    for (int e = 0; e < 16; ++e) hv[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
                    uint4 *d = reinterpret_cast<uint4 *>(a.dz + (r0 + r) * kTrainCh);
                    #pragma unroll
                    for (int e = 0; e < 4; ++e)
                        d[e] = make_uint4(hv[4 * e], hv[4 * e + 1], hv[4 * e + 2], hv[4 * e + 3]);
                }
            } else {
                // weight gradients: lane = hidden unit
                for (int mt = 0; mt < 2; ++mt) {
                    const int n = 128 * mt + 32 * (warp & 3) + lane;
                    float v[32];
                    tmem_ld32(tq + kDw1 + uint32_t(32 * mt), v);
                    #pragma unroll
                    for (int e = 0; e < 8; ++e)
                        *reinterpret_cast<float4 *>(smem + S::kDa + (n * 36 + 4 * e) * 4) =
                            make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                    tmem_ld16(tq + kDw2 + uint32_t(16 * mt), v);
                    #pragma unroll
                    for (int d = 0; d < DIM; ++d) p_w2[d * kHid + n] = v[d];
                }
            }
            fence_before();
            __syncthreads();
            if (tid < kTrainCh) {
                float s = 0.f;
                for (int r = 0; r < a.R; ++r) s += st[r * 33 + tid];
                p_db[tid] = s;
            }
            for (int i = tid; i < kHid * kTrainCh; i += 256)
                part[i] = reinterpret_cast<const float *>(smem + S::kDa)[(i >> 5) * 36 + (i & 31)];
        }
    }
    mma_drain(bars + 2, tmem, kCols, warp);
}

// ---------------------------------------------------------------------------
// Sums of the CTAs' partials in a fixed order. Few partials (up to kRedFew):
// a thread adds them all, four neighbouring elements at a time where the
// alignment allows. Many: 32 elements per block, eight groups of threads take
// every eighth partial each and their sums are added in order (a long chain of
// loads per thread would be latency alone). Loads are issued eight at a time: one
// after the other the classifier's sums took 71 us, now 15.
// ---------------------------------------------------------------------------
constexpr int kRedE = 32, kRedG = 8, kRedFew = 48, kRedT = kRedE * kRedG;

struct ReduceArgs {
    ReduceSeg seg[kMaxSegs];
    int block0[kMaxSegs + 1];
    int vec[kMaxSegs];            // elements per thread of a segment of few, else 0
    int n;
};

__device__ __forceinline__ void reduce_store(const ReduceSeg &g, int64_t i, float v) {
    g.out[i] = g.div > 0.f ? v / g.div : v;
}

__global__ void __launch_bounds__(kRedT) reduce_parts_kernel(const ReduceArgs a) {
    __shared__ float red[kRedG][kRedE];
    int s = 0;
    while (s + 1 < a.n && int(blockIdx.x) >= a.block0[s + 1]) ++s;
    const ReduceSeg &g = a.seg[s];
    const int64_t blk = blockIdx.x - a.block0[s];
    pdl_wait();
    // batches of loads in flight together, then added in order
    constexpr int kBatch = 8;
    if (a.vec[s] == 4) {
        const int64_t i = (blk * kRedT + threadIdx.x) * 4;
        if (i >= g.count) return;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q0 = 0; q0 < g.n; q0 += kBatch) {
            float4 v[kBatch];
            #pragma unroll
            for (int j = 0; j < kBatch; ++j)
                v[j] = q0 + j < g.n ? __ldg(reinterpret_cast<const float4 *>(
                                          g.part + int64_t(q0 + j) * g.stride + i))
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
            #pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                x.x += v[j].x;
                x.y += v[j].y;
                x.z += v[j].z;
                x.w += v[j].w;
            }
        }
        reduce_store(g, i, x.x);
        reduce_store(g, i + 1, x.y);
        reduce_store(g, i + 2, x.z);
        reduce_store(g, i + 3, x.w);
        return;
    }
    const bool few = a.vec[s] == 1;
    const int e = threadIdx.x % kRedE, grp = threadIdx.x / kRedE;
    const int64_t i = few ? blk * kRedT + threadIdx.x : blk * kRedE + e;
    float x = 0.f;
    if (i < g.count) {
        const int step = few ? 1 : kRedG;
        for (int q0 = few ? 0 : grp; q0 < g.n; q0 += step * kBatch) {
            float v[kBatch];
            #pragma unroll
            for (int j = 0; j < kBatch; ++j)
                v[j] = q0 + j * step < g.n ? __ldg(g.part + int64_t(q0 + j * step) * g.stride + i) : 0.f;
            #pragma unroll
            for (int j = 0; j < kBatch; ++j) x += v[j];
        }
    }
    if (few) {
        if (i < g.count) reduce_store(g, i, x);
        return;
    }
    red[grp][e] = x;
    __syncthreads();
    if (grp == 0 && i < g.count) {
        float v = red[0][e];
        #pragma unroll
        for (int q = 1; q < kRedG; ++q) v += red[q][e];
        reduce_store(g, i, v);
    }
}

// the kernels' instances: f(Geo) for the layer's dimension and edge
template <class Fn>
void with_geo(const ConvGeo &g, bool first, Fn f) {
    if (g.dim == 2) {
        if (first) {
            if (g.Si == 9) f(Geo<2, 9, true>());          // regressor
            if (g.Si == 11) f(Geo<2, 11, true>());        // classifier, zero ring stored
        } else {
            if (g.Si == 11) f(Geo<2, 11, false>());
            if (g.Si == 7) f(Geo<2, 7, false>());
            if (g.Si == 5) f(Geo<2, 5, false>());
            if (g.Si == 3) f(Geo<2, 3, false>());
        }
    } else if (first) {
        if (g.Si == 7) f(Geo<3, 7, true>());
    } else {
        if (g.Si == 5) f(Geo<3, 5, false>());
        if (g.Si == 3) f(Geo<3, 3, false>());
    }
}

// inputs per tile of the im2col kernels: as many as fill the 128 rows and fit
// shared memory, but no more than leaves every SM a tile
template <class N, bool BWD>
int tile_inputs(int64_t B, int sm_count) {
    const int64_t even = (B + sm_count - 1) / sm_count;
    int G = int(std::max<int64_t>(1, std::min<int64_t>(N::GMax, even)));
    while (G > 1 && conv_smem<N, BWD>(G).total > kSmemMax) --G;
    return G;
}

// inputs per tile of the backward pass: the same number of tiles for every SM (a
// tile's time hardly falls with its inputs, so 4096 rows of Si = 5 run as three
// tiles of 9 per SM, not as 2.7 of 10)
template <class N>
int bwd_inputs(int64_t B, int sm_count) {
    const int64_t each = int64_t(sm_count) * BwdCfg<N>::GMax, rounds = (B + each - 1) / each;
    return int((B + sm_count * rounds - 1) / (sm_count * rounds));
}

int head_rows(int64_t B, int sm_count) {
    return B <= int64_t(32) * sm_count ? 32 : B <= int64_t(64) * sm_count ? 64 : 128;
}

}  // namespace

int train_packed_kw(int dim) { return kTrainCh * (dim == 2 ? 9 : 27); }

int launch_pack_train(const PackSeg *segs, int n, cudaStream_t st) {
    PackArgs a{};
    a.n = n;
    for (int i = 0; i < n; ++i) a.seg[i] = segs[i];
    launch_pdl(pack_train_kernel, dim3(76), dim3(256), 0, st, a);
    return 1;
}

int launch_conv_fwd(const ConvGeo &g, const void *x, bool first, int64_t B, const uint8_t *packed,
                    const float *bias, uint16_t *y, int ring, float *z, int *err, int sm_count,
                    cudaStream_t st) {
    ConvArgs a{};
    a.x = x;
    a.B = B;
    a.w = packed;
    a.bias = bias;
    a.y = y;
    a.z = z;
    a.ring = ring;
    // the general GEMM's K splits of this product (tc_gemm.cu): the same
    // partial sums give the same bits
    const int64_t chunks = (g.K + 63) / 64, tiles = (B * g.Po + 127) / 128;
    int64_t splits = 1;
    if (tiles < 2 * sm_count && chunks > 8)
        splits = std::min<int64_t>(chunks / 4, (2 * sm_count + tiles - 1) / tiles);
    a.kc = int((chunks + splits - 1) / splits * 64);
    a.nsplit = (g.K + a.kc - 1) / a.kc;
    with_geo(g, first, [&](auto n) {
        using N = decltype(n);
        a.G = tile_inputs<N, false>(B, sm_count);
        a.tiles = (B + a.G - 1) / a.G;
        const ConvSmem L = conv_smem<N, false>(a.G);
        cudaFuncSetAttribute(conv_fwd_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        const int per_sm = L.total <= kSmemHalf ? 2 : 1;
        const int grid = int(std::min<int64_t>(a.tiles, int64_t(sm_count) * per_sm));
        launch_pdl(conv_fwd_kernel<N>, dim3(grid), dim3(kFwdThreads), size_t(L.total), st, a, L, err);
    });
    return 1;
}

int conv_bwd_ctas(const ConvGeo &g, int64_t B, bool first, int sm_count) {
    int64_t ctas = 1;
    with_geo(g, first, [&](auto n) {
        using N = decltype(n);
        if constexpr (N::First) {
            const int G = tile_inputs<N, true>(B, sm_count);
            ctas = std::min<int64_t>((B + G - 1) / G, int64_t(sm_count) * ConvCfg<N, true>::PerSm);
        } else {
            const int G = bwd_inputs<N>(B, sm_count);
            ctas = std::min<int64_t>((B + G - 1) / G, sm_count);
        }
    });
    return int(ctas);
}

int launch_conv_bwd(const ConvGeo &g, const void *x, bool first, int64_t B, const uint16_t *dz,
                    const uint8_t *packed, float *wpart, uint16_t *dzp, float *bpart, int *err,
                    int sm_count, cudaStream_t st) {
    ConvArgs a{};
    a.x = x;
    a.B = B;
    a.w = packed;
    a.dz = dz;
    a.wpart = wpart;
    a.dzp = dzp;
    a.bpart = bpart;
    const int grid = conv_bwd_ctas(g, B, first, sm_count);
    with_geo(g, first, [&](auto n) {
        using N = decltype(n);
        if constexpr (N::First) {
            a.G = tile_inputs<N, true>(B, sm_count);
            a.tiles = (B + a.G - 1) / a.G;
            const ConvSmem L = conv_smem<N, true>(a.G);
            static_assert(ConvCfg<N, true>::PerSm == 1 || conv_smem<N, true>(1).total <= kSmemHalf,
                          "two CTAs per SM");
            cudaFuncSetAttribute(first_wgrad_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
            launch_pdl(first_wgrad_kernel<N>, dim3(grid), dim3(kWgThreads), size_t(L.total), st, a, L, err);
        } else {
            using F = BwdCfg<N>;
            a.G = bwd_inputs<N>(B, sm_count);
            a.tiles = (B + a.G - 1) / a.G;
            cudaFuncSetAttribute(conv_bwd_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, F::kTotal);
            launch_pdl(conv_bwd_kernel<N>, dim3(grid), dim3(kBwdThreads), size_t(F::kTotal), st, a, err);
        }
    });
    return 1;
}

int head_ctas(int64_t B, int sm_count) {
    const int R = head_rows(B, sm_count);
    return int((B + R - 1) / R);
}

int64_t head_part_floats(int dim) {
    return kHid * kTrainCh + kHid + dim * kHid + dim + kTrainCh + 1;
}

int launch_train_head(int dim, int64_t B, const uint16_t *h, const uint8_t *packed_w1,
                      const float *b1, const float *W2, const float *b2, const float *tgt,
                      float *out, uint16_t *dz, float *part, int *err, int sm_count,
                      cudaStream_t st) {
    HeadArgs a{B, head_rows(B, sm_count), h, packed_w1, b1, W2, b2, tgt, out, dz, part};
    const int grid = head_ctas(B, sm_count);
    auto *k = dim == 2 ? head_train_kernel<2> : head_train_kernel<3>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, HeadSmem::kTotal);
    launch_pdl(k, dim3(grid), dim3(256), size_t(HeadSmem::kTotal), st, a, err);
    return 1;
}

int launch_reduce_parts(const ReduceSeg *segs, int n_segs, cudaStream_t st) {
    ReduceArgs a{};
    a.n = n_segs;
    int blocks = 0;
    for (int s = 0; s < n_segs; ++s) {
        const ReduceSeg &g = a.seg[s] = segs[s];
        const bool four = g.count % 4 == 0 && g.stride % 4 == 0 &&
                          (reinterpret_cast<uintptr_t>(g.part) & 15u) == 0;
        a.vec[s] = g.n > kRedFew ? 0 : four ? 4 : 1;
        a.block0[s] = blocks;
        const int per = a.vec[s] ? kRedT * a.vec[s] : kRedE;
        blocks += int((g.count + per - 1) / per);
    }
    a.block0[n_segs] = blocks;
    launch_pdl(reduce_parts_kernel, dim3(blocks), dim3(kRedT), 0, st, a);
    return 1;
}

}  // namespace cs
