// Module 1 of the classifier predictor (Sec. 2.3) fused on the tensor cores:
// the pooled-centroid window of a particle, its two zero-padded 3^D
// convolutions of 32 channels with ReLU and the 2^D average pooling, in one
// CTA, with no im2col copy and no activation leaving shared memory.
//
// Layout. A particle's window with its zero padding sits on a flat index
// q = (z E + y) E + x of pitch E = W + 1: the ring's cells before a line are
// the ring's cells after the line before it (and so for planes, and for the
// next particle of a group), so one zero column and row serve both. A
// convolution output is computed at the row r = q - (E + 1) (2-D;
// q - (E^2 + E + 1) in 3-D) of the window position q it belongs to, and reads
// its input at r + shift(tap), shift = (dz E + dy) E + dx: a tap is a row
// offset of the shared-memory operand, so each convolution is an implicit
// GEMM. Output rows whose position lies outside the window (the ring's
// columns) are garbage and are never stored or pooled. In 2-D a group of NP = 5
// particles (100 rows each) fills four M-tiles of 128 rows, where a particle
// on its own takes one; in 3-D a particle takes four (five at pitch W + 2).
//
//   input  [rows][8] BF16: the D window channels and 8 - D zero channels;
//          the ring and the rows past the window stay zero
//   conv1  tcgen05.mma kind::f16, M = 128 rows, N = 32, K = 16 = two taps of
//          8 channels: the A descriptor's leading byte offset is the row
//          distance of the two taps (5 MMAs per M-tile in 2-D, 14 in 3-D). The
//          odd last tap's partner is a block of zero rows with zero weights: rows
//          of the window there would turn an infinite input into a NaN
//   conv2  K = 32 channels of one tap in two K = 16 steps: 2 MMAs per tap
//   act    [4 chunks][rows][8] BF16: ReLU(conv1 + b1), written at the window
//          position of each valid output row (its padded layout is conv2's
//          operand, ring zero)
//   stage  [pooled positions][33] FP32: ReLU(conv2 + b2), read by the pooling
//   FP32 accumulation in TMEM: conv1 in columns [0, 32 MT), conv2 in the next
//   range of 32 MT (or two, by turns), MT the M-tiles of a group.
// An MMA of M = 128, N = 32, K = 16 takes 42 cycles whatever its row offset,
// if it is issued as fast: the taps are unrolled, so that issuing one is a
// few additions to a descriptor (with the taps in a loop it took 58).
//
// Inputs. Each window cell holds (p - x_p) / s: p is the cell's pooled
// element centroid, given as float hi + lo parts, so the difference is taken
// in FP32 to about one unit in the last place of the FP64 value; a cell
// outside the grid or without a centroid holds its centre, (e - W/2) - offset
// in cell units. x_p's cell is the FP64 formula's (certified in FP32, with the
// FP64 formula as arbiter: the same cell as the labels and the start rule);
// its offset from the cell centre is taken in FP32.
//
// Pipeline. Warps 0-7 compute the inputs and run conv1's epilogue, warps 8-15
// in 3-D (the same warps in 2-D) conv2's epilogue and the pooling: warp w reads
// TMEM lanes 32 (w % 4) .. and 16 of the 32 channels. One more warp issues the
// MMAs. A CTA takes groups blockIdx.x, blockIdx.x + gridDim.x, ... In 3-D
// inputs, activations and conv2's accumulators have two buffers (NB), and conv1
// of group k + 1 is issued before conv2 of group k: while conv2(k) holds the
// tensor pipe, conv1(k + 1)'s epilogue, the inputs of k + 3 and conv2(k - 1)'s
// epilogue run. In 2-D, where a group's inputs and epilogues take about as long
// as its products, two CTAs per SM with one buffer each overlap better. Every
// wait is bounded; one that gives up raises the CTA's abort flag and the device
// error flag.
//
// Bound by the tensor pipe's rate at N = 32 in 3-D (272 MMAs of 42 cycles a
// particle: 648 us per chunk of 16384 at 152 SMs and 1.9 GHz), by the epilogues
// and inputs in 2-D (92 MMAs a group of five: 88 us per chunk of 32768).
// Measured: 662 us and 127 us. One set of warps for both epilogues and one
// buffer: 807 us in 3-D; two buffers and one CTA per SM: 158 us in 2-D, two
// sets and two CTAs 131 us. Padded by W + 2, one particle a group, with taps in a
// loop: 1045 us and 182 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "classifier.h"
#include "launch_attr.h"
#include "tc_common.cuh"

namespace cs {
namespace {

constexpr int kEpiC = 8;                    // warps of an epilogue set

template <int D, int NP_>
struct ClsGeo {
    static constexpr int NP = NP_;                                   // particles of a group
    static constexpr int NB = D == 3 ? 2 : 1;                        // buffers
    static constexpr int Sets = D == 3 ? 2 : 1;                      // epilogue sets
    static constexpr int PerSm = D == 3 ? 1 : NP_ > 1 ? 2 : 3;       // CTAs per SM
    static constexpr int MmaWarp = Sets * kEpiC;                     // issues the MMAs
    static constexpr int Threads = (MmaWarp + 1) * 32;
    static_assert(D == 2 || NP == 1, "groups of particles in 2-D only");
    static constexpr int W = D == 2 ? 9 : 7;
    static constexpr int E = W + 1;                                  // pitch
    static constexpr int P = D == 2 ? W * W : W * W * W;             // window cells
    static constexpr int Pitch = D == 2 ? E * E : E * E * E;         // rows of a particle
    static constexpr int S = D == 2 ? 2 * E + 2 : (2 * E + 2) * E + 2;   // largest tap shift
    static constexpr int Ro = (NP - 1) * Pitch +
                              (D == 2 ? (W - 1) * E + W : ((W - 1) * E + W - 1) * E + W);
    static constexpr int MT = (Ro + 127) / 128;                      // M-tiles per group
    static constexpr int Rows = (128 * MT + S + 8 + 7) / 8 * 8;      // operand rows
    static constexpr int Coff = D == 2 ? E + 1 : (E + 1) * E + 1;    // output row -> position
    static constexpr int Taps = D == 2 ? 9 : 27;
    static constexpr int Pairs = (Taps + 1) / 2;
    static constexpr int Wp = W / 2;
    static constexpr int Pp = D == 2 ? Wp * Wp : Wp * Wp * Wp;
    static constexpr int Ws = 2 * Wp;                                // edge that is pooled
    static constexpr int Ps = D == 2 ? Ws * Ws : Ws * Ws * Ws;
    static constexpr int Ld = 33;                                    // stage row stride (floats)
    static constexpr int NeedCols = 32 * MT * (1 + NB);
    static constexpr uint32_t Cols = NeedCols <= 64 ? 64 : NeedCols <= 128 ? 128 : NeedCols <= 256 ? 256 : 512;
    // packed weights
    static constexpr int kW1 = 0;                                    // bf16 [Pairs][2][32][8]
    static constexpr int kB1 = kW1 + Pairs * 1024;                   // f32 [32]
    static constexpr int kW2 = kB1 + 128;                            // bf16 [Taps][4][32][8]
    static constexpr int kB2 = kW2 + Taps * 2048;                    // f32 [32]
    static constexpr int kPacked = kB2 + 128;
    // shared memory
    static constexpr int kSmZero = 0;                                // 128 zero rows
    static constexpr int kSmIn = kSmZero + 128 * 16;
    static constexpr int kSmAct = kSmIn + NB * Rows * 16;
    static constexpr int kSmW = kSmAct + NB * 4 * Rows * 16;
    static constexpr int kSmStage = kSmW + kPacked;
    static constexpr int kSmBar = (kSmStage + NP * Ps * Ld * 4 + 7) / 8 * 8;   // mbarriers [4]
    static constexpr int kSmCnt = kSmBar + 4 * 8;                    // u32 in_ready, act_ready, out_free
    // per particle: int c0[3], float off[3], x hi/lo [6]
    static constexpr int kSmPart = kSmCnt + 16;
    static constexpr int kSmSlot = kSmPart + NP * 12 * 4;            // TMEM address, abort flag
    static constexpr int kSmTotal = kSmSlot + 16;

    static_assert(NeedCols <= int(Cols) && int(Cols) * PerSm <= 512, "TMEM columns");
    static_assert(128 * MT + S < Rows, "operand reads in bounds");
    static_assert(Ro - 1 + Coff < Rows, "outputs land in the window");
    static_assert(kSmTotal <= (PerSm == 1 ? 232448 : PerSm == 2 ? 113 * 1024 : 75 * 1024), "shared memory of one CTA");
    static_assert(kSmW % 128 == 0 && kSmAct % 128 == 0, "operand alignment");
};

template <int D>
__device__ __forceinline__ constexpr int cls_shift(int t) {
    constexpr int E = ClsGeo<D, 1>::E;
    return D == 2 ? (t / 3) * E + t % 3 : ((t / 9) * E + (t / 3) % 3) * E + t % 3;
}

// named barrier `id` (1, 2) over a set of epilogue warps
__device__ __forceinline__ void epi_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kEpiC * 32) : "memory");
}
__device__ __forceinline__ bool epi_or(int id, bool flag) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, %3, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(r)
        : "r"(uint32_t(flag)), "n"(kEpiC * 32), "r"(id)
        : "memory");
    return r != 0;
}

// x_p's ASG cell on axis k and its offset from the cell centre (cell units).
// The cell is the FP64 formula's (floor((x - lo) / s), clamped): taken in
// FP32 from x's hi + lo parts where the rounding bound cannot move the
// quotient across an integer, else by the FP64 formula itself (the
// certification of the walk's cell indices). The offset is the FP32
// quotient minus (cell + 1/2), within ~1e-7 of the quotient of the FP64 one.
__device__ __forceinline__ void cell_offset(const DevMesh &m, int k, double x, float xh, float xl,
                                            int &cell, float &off) {
    const float df = (xh - m.lo_h[k]) + (xl - m.lo_l[k]);
    const float ed = delta_bound(df, xh, m.lo_h[k]);
    const float q = df * m.inv_sa[k];
    const float bnd = fmaf(2.0f * ed, m.inv_sa[k], fmaf(k8U, fabsf(q), kTiny));
    const int a = __float2int_rd(q - bnd), b = __float2int_rd(q + bnd);
    int64_t i;
    if (a == b && fabsf(q) < 4.0e6f)
        i = a < 0 ? 0 : (a > m.ga[k] - 1 ? m.ga[k] - 1 : a);
    else
        i = cell_axis64(x, m.lo[k], m.sa[k], m.ga[k]);
    cell = int(i);
    off = q - (float(i) + 0.5f);
}

// The inputs of particles [b0, b0 + nb) into the operand rows (epilogue
// warps): thread tid < nb D first computes an axis's cell, offset and the
// hi/lo split of x_p; then every window cell is one 16-byte row.
template <int D, int NP>
__device__ __forceinline__ void cls_inputs(const DevMesh &m, const float *__restrict__ pool_f,
                                           const double *__restrict__ xp, int64_t b0, int nb,
                                           uint8_t *in, float *part, float *__restrict__ off_out,
                                           int tid) {
    using G = ClsGeo<D, NP>;
    if (tid < nb * D) {
        const int w = tid / D, k = tid % D;
        float *sp = part + 12 * w;
        const double x = xp[b0 * D + tid];
        const float h = __double2float_rn(x);
        const float l = __double2float_rn(__dsub_rn(x, double(h)));
        int c0 = 0;
        float o = 0.f;
        #pragma unroll
        for (int q = 0; q < D; ++q)
            if (k == q) cell_offset(m, q, x, h, l, c0, o);
        reinterpret_cast<int *>(sp)[k] = c0;
        sp[3 + k] = o;
        off_out[b0 * D + tid] = o;
        sp[6 + k] = h;
        sp[9 + k] = l;
    }
    epi_sync(1);
    for (int i = tid; i < nb * G::P; i += kEpiC * 32) {
        const int w = i / G::P, e = i % G::P;
        const float *sp = part + 12 * w;
        int ek[3] = {e % G::W, (e / G::W) % G::W, D == 3 ? e / (G::W * G::W) : 0};
        bool inside = true;
        int64_t flat = 0;
        int cc[3];
        #pragma unroll
        for (int k = 0; k < D; ++k) {
            cc[k] = reinterpret_cast<const int *>(sp)[k] - G::W / 2 + ek[k];
            inside &= cc[k] >= 0 && cc[k] < m.ga[k];
        }
        #pragma unroll
        for (int k = D - 1; k >= 0; --k) flat = flat * m.ga[k] + (inside ? cc[k] : 0);
        float v[3] = {0.f, 0.f, 0.f};
        bool has = false;
        float ph[3], pl[3];
        if (inside) {
            if constexpr (D == 2) {
                const float4 q = __ldg(reinterpret_cast<const float4 *>(pool_f) + flat);
                ph[0] = q.x;
                pl[0] = q.y;
                ph[1] = q.z;
                pl[1] = q.w;
            } else {
                #pragma unroll
                for (int k = 0; k < D; ++k) {
                    const float2 q = __ldg(reinterpret_cast<const float2 *>(pool_f) + flat * D + k);
                    ph[k] = q.x;
                    pl[k] = q.y;
                }
            }
            has = !isnan(ph[0]);
        }
        #pragma unroll
        for (int k = 0; k < D; ++k) {
            const float inv = m.inv_sa[k];
            v[k] = has ? __fmul_rn(__fadd_rn(__fsub_rn(ph[k], sp[6 + k]), __fsub_rn(pl[k], sp[9 + k])),
                                   inv)
                       : __fsub_rn(float(ek[k] - G::W / 2), sp[3 + k]);
        }
        const int q = w * G::Pitch + (D == 2 ? (ek[1] + 1) * G::E + ek[0] + 1
                                             : ((ek[2] + 1) * G::E + ek[1] + 1) * G::E + ek[0] + 1);
        *reinterpret_cast<uint4 *>(in + 16 * q) =
            make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], 0.f), 0u, 0u);
    }
}

template <int D, int NP>
__global__ void __launch_bounds__(ClsGeo<D, NP>::Threads, ClsGeo<D, NP>::PerSm) cls_conv_tc_kernel(
    const DevMesh m, const float *__restrict__ pool_f, int64_t B, const double *__restrict__ xp,
    const uint8_t *__restrict__ packed, const FcMat cat, float *__restrict__ off_out, int *err) {
    using G = ClsGeo<D, NP>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *in = smem + G::kSmIn;
    uint8_t *act = smem + G::kSmAct;
    uint8_t *wsm = smem + G::kSmW;
    float *stage = reinterpret_cast<float *>(smem + G::kSmStage);
    // conv1; conv2, one per buffer; final
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + G::kSmBar);
    // groups whose inputs are in place; whose conv1 epilogue is done; whose conv2
    // accumulators are read
    uint32_t *in_ready = reinterpret_cast<uint32_t *>(smem + G::kSmCnt);
    uint32_t *act_ready = in_ready + 1, *out_free = in_ready + 2;
    float *part = reinterpret_cast<float *>(smem + G::kSmPart);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + G::kSmSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + G::kSmSlot + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // operands zero (ring, padding channels, rows past the window), barriers, TMEM
    for (int i = tid; i < G::kSmW / 16; i += G::Threads)
        reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(bars + i, 1u);
        *in_ready = 0;
        *act_ready = 0;
        *out_free = 0;
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(tmem_slot)),
                     "r"(G::Cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (int i = tid; i < G::kPacked / 16; i += G::Threads) cp_async16(wsm + 16 * i, packed + 16 * i);
    cp_async_wait_all();
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int64_t groups = (B + NP - 1) / NP;
    const int n_mine = groups > blockIdx.x ? int((groups - 1 - blockIdx.x) / gridDim.x + 1) : 0;
    const int wq = warp & 3, c0 = 16 * ((warp & 7) >> 2);     // lane quarter, first channel
    const uint32_t tq = tmem + (uint32_t(32 * wq) << 16) + uint32_t(c0);

    if (warp == G::MmaWarp) {
        const bool leader = elect_one();
        const uint64_t d_w1 = sdesc(smem_addr(wsm + G::kW1), 32 * 16, 128);
        const uint64_t d_w2 = sdesc(smem_addr(wsm + G::kW2), 32 * 16, 128);
        constexpr uint32_t id32 = idesc_bf16(128, 32);
        auto conv1 = [&](int k) {
            const uint64_t d_in = sdesc(smem_addr(in + (k % G::NB) * G::Rows * 16), 0, 128);
            // the zero rows, and the distance to the buffer's last tap from there
            const uint64_t d_zero = sdesc(smem_addr(smem + G::kSmZero),
                                          G::kSmIn + (k % G::NB) * G::Rows * 16 + cls_shift<D>(G::Taps - 1) * 16, 128);
            #pragma unroll 1
            for (int mt = 0; mt < G::MT; ++mt) {
                const uint32_t dcol = tmem + uint32_t(32 * mt);
                #pragma unroll
                for (int i = 0; i < G::Pairs; ++i) {
                    const int sh0 = cls_shift<D>(2 * i);
                    const int sh1 = cls_shift<D>(i + 1 < G::Pairs ? 2 * i + 1 : 2 * i);
                    const uint64_t a = i + 1 < G::Pairs
                                           ? d_in + uint64_t(128 * mt + sh0) + (uint64_t(sh1 - sh0) << 16)
                                           : d_zero + (uint64_t(128 * mt) << 16);
                    mma_bf16(dcol, a, d_w1 + uint64_t(i * 64), id32, i > 0 ? 1u : 0u);
                }
            }
            mma_commit(bars + 0);
        };
        auto conv2 = [&](int k) {
            const uint64_t d_act = sdesc(smem_addr(act + (k % G::NB) * 4 * G::Rows * 16), G::Rows * 16, 128);
            #pragma unroll 1
            for (int mt = 0; mt < G::MT; ++mt) {
                const uint32_t dcol = tmem + uint32_t(32 * (G::MT * (1 + k % G::NB) + mt));
                // nine taps unrolled, a plane (3-D) at a time: more of them hold
                // their offsets in more registers than there are
                #pragma unroll 1
                for (int tz = 0; tz < G::Taps / 9; ++tz) {
                    const uint64_t az = d_act + uint64_t(128 * mt + tz * G::E * G::E);
                    const uint64_t wz = d_w2 + uint64_t(tz * 9 * 4 * 32);
                    #pragma unroll
                    for (int t = 0; t < 9; ++t)
                        #pragma unroll
                        for (int kk = 0; kk < 2; ++kk)
                            mma_bf16(dcol, az + uint64_t(2 * kk * G::Rows + (t / 3) * G::E + t % 3),
                                     wz + uint64_t((t * 4 + 2 * kk) * 32), id32,
                                     (tz | t | kk) != 0 ? 1u : 0u);
                }
            }
            mma_commit(bars + 1 + k % G::NB);
        };
        bool ok = n_mine == 0 || wait_count(in_ready, 1u, abort_flag, err);
        fence_after();
        if (ok && n_mine > 0 && leader) conv1(0);
        __syncwarp();
        for (int k = 0; k < n_mine && ok; ++k) {
            // conv1's accumulators are read and its activations written; the
            // accumulators that conv2 takes are read
            ok = wait_count(act_ready, uint32_t(k + 1), abort_flag, err);
            if (G::Sets == 2 && ok && k >= G::NB) ok = wait_count(out_free, uint32_t(k - G::NB + 1), abort_flag, err);
            if (ok && G::NB == 2 && k + 1 < n_mine)
                ok = wait_count(in_ready, uint32_t(k + 2), abort_flag, err);
            if (!ok) break;
            fence_after();
            if (leader) {
                if (G::NB == 2 && k + 1 < n_mine) conv1(k + 1);
                conv2(k);
            }
            __syncwarp();
            if (G::NB == 1 && k + 1 < n_mine) {
                ok = wait_count(in_ready, uint32_t(k + 2), abort_flag, err);
                if (!ok) break;
                fence_after();
                if (leader) conv1(k + 1);
                __syncwarp();
            }
        }
    } else {
        const float *b1 = reinterpret_cast<const float *>(wsm + G::kB1);
        const float *b2 = reinterpret_cast<const float *>(wsm + G::kB2);
        auto inputs = [&](int k) {
            const int64_t b0 = (blockIdx.x + int64_t(k) * gridDim.x) * NP;
            cls_inputs<D, NP>(m, pool_f, xp, b0, int(min(int64_t(NP), B - b0)),
                              in + (k % G::NB) * G::Rows * 16, part, off_out, tid);
            fence_async_smem();
            epi_sync(1);
            if (tid == 0) red_release_add(in_ready, 1u);
        };
        auto epilogue1 = [&](int k) {
            // ---- conv1 epilogue: ReLU(z + b1) in BF16 at each valid row's window
            //      position, once conv2(k - NB) has read that buffer ----
            bool ok = __all_sync(kFull, mbar_wait(bars + 0, uint32_t(k & 1), abort_flag, err)) != 0;
            if (ok && k >= G::NB)
                ok = __all_sync(kFull, mbar_wait(bars + 1 + k % G::NB, uint32_t(k / G::NB - 1) & 1u,
                                                 abort_flag, err)) != 0;
            if (epi_or(1, !ok)) return false;
            fence_after();
            uint8_t *ak = act + (k % G::NB) * 4 * G::Rows * 16 + (size_t(c0 >> 3) * G::Rows + G::Coff) * 16;
            for (int mt = 0; mt < G::MT; ++mt) {
                float v[16];
                tmem_ld16(tq + uint32_t(32 * mt), v);
                uint32_t hv[8];
                bias_relu_bf16_16(v, b1 + c0, hv);
                const int r = 128 * mt + 32 * wq + lane;
                const int rr = r % G::Pitch;
                const int x = rr % G::E, y = (rr / G::E) % G::E, z = D == 3 ? rr / (G::E * G::E) : 0;
                if (r < G::Ro && x < G::W && y < G::W && z < G::W) {
                    uint8_t *o = ak + r * 16;
                    *reinterpret_cast<uint4 *>(o) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
                    *reinterpret_cast<uint4 *>(o + G::Rows * 16) = make_uint4(hv[4], hv[5], hv[6], hv[7]);
                }
            }
            fence_before();
            fence_async_smem();
            epi_sync(1);
            if (tid == 0) red_release_add(act_ready, 1u);
            return true;
        };
        constexpr int kBar2 = G::Sets;
        const int t2 = tid - (G::Sets - 1) * kEpiC * 32;
        auto epilogue2 = [&](int k) {
            const int64_t b0 = (blockIdx.x + int64_t(k) * gridDim.x) * NP;
            const int nb = int(min(int64_t(NP), B - b0));
            // ---- conv2 epilogue: ReLU(z + b2) in FP32 to the stage, then pooling ----
            const bool ok = __all_sync(kFull, mbar_wait(bars + 1 + k % G::NB, uint32_t(k / G::NB) & 1u,
                                                        abort_flag, err)) != 0;
            if (epi_or(kBar2, !ok)) return false;
            fence_after();
            for (int mt = 0; mt < G::MT; ++mt) {
                float v[16];
                tmem_ld16(tq + uint32_t(32 * (G::MT * (1 + k % G::NB) + mt)), v);
                const int r = 128 * mt + 32 * wq + lane, w = r / G::Pitch, rr = r % G::Pitch;
                const int x = rr % G::E, y = (rr / G::E) % G::E, z = D == 3 ? rr / (G::E * G::E) : 0;
                if (r < G::Ro && x < G::Ws && y < G::Ws && z < G::Ws) {
                    float *st = stage + (w * G::Ps + (z * G::Ws + y) * G::Ws + x) * G::Ld + c0;
                    #pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float4 b = *reinterpret_cast<const float4 *>(b2 + c0 + 4 * e);
                        st[4 * e] = fmaxf(v[4 * e] + b.x, 0.f);
                        st[4 * e + 1] = fmaxf(v[4 * e + 1] + b.y, 0.f);
                        st[4 * e + 2] = fmaxf(v[4 * e + 2] + b.z, 0.f);
                        st[4 * e + 3] = fmaxf(v[4 * e + 3] + b.w, 0.f);
                    }
                }
            }
            fence_before();
            epi_sync(kBar2);
            if (G::Sets == 2 && t2 == 0) red_release_add(out_free, 1u);
            // BF16 into the tiled feature matrix (fc_tc.h): column c Pp + pp of
            // the particle's row. 2-D: four neighbouring columns per thread
            constexpr int kPer = G::Pp % 4 == 0 ? 4 : 1, kUnits = 32 * G::Pp / kPer;
            for (int i = t2; i < nb * kUnits; i += kEpiC * 32) {
                const int w = i / kUnits, u0 = i % kUnits, c = u0 % 32, p0 = u0 / 32 * kPer;
                const float *st = stage + w * G::Ps * G::Ld + c;
                float s[kPer];
                #pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int pp = p0 + u;
                    const int px = pp % G::Wp, py = (pp / G::Wp) % G::Wp, pz = D == 3 ? pp / (G::Wp * G::Wp) : 0;
                    s[u] = 0.f;
                    #pragma unroll
                    for (int oz = 0; oz < (D == 3 ? 2 : 1); ++oz)
                        #pragma unroll
                        for (int oy = 0; oy < 2; ++oy)
                            #pragma unroll
                            for (int ox = 0; ox < 2; ++ox)
                                s[u] += st[(((2 * pz + oz) * G::Ws + 2 * py + oy) * G::Ws + 2 * px + ox) * G::Ld];
                    s[u] = s[u] / float(1 << D);
                }
                const int col = c * G::Pp + p0;
                const int64_t b = b0 + w;
                uint8_t *o = cat.p + (b >> 7) * cat.tile + int64_t(cat.chunk0 + (col >> 3)) * kFcChunk +
                             (b & 127) * 16 + (col & 7) * 2;
                if constexpr (kPer == 4)
                    *reinterpret_cast<uint2 *>(o) =
                        make_uint2(pack_bf16x2(s[0], s[1]), pack_bf16x2(s[2], s[3]));
                else
                    *reinterpret_cast<__nv_bfloat16 *>(o) = __float2bfloat16_rn(s[0]);
            }
            epi_sync(kBar2);      // the stage is free
            return true;
        };
        if (warp < kEpiC) {
            for (int k = 0; k < G::NB && k < n_mine; ++k) inputs(k);
            for (int k = 0; k < n_mine && epilogue1(k); ++k) {
                // conv1(k) has read its inputs' buffer
                if (k + G::NB < n_mine) inputs(k + G::NB);
                if (G::Sets == 1 && !epilogue2(k)) break;
            }
        } else {
            for (int k = 0; k < n_mine && epilogue2(k); ++k) {}
        }
    }
    // wait (bounded) for this CTA's MMAs in flight before TMEM is released
    if (warp == G::MmaWarp) {
        if (elect_one()) {
            mma_commit(bars + 3);
            for (uint32_t i = 0; i < (1u << 24) && !mbar_try_wait(bars + 3, 0); ++i)
                if (i > 64) __nanosleep(64);
        }
        __syncwarp();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G::Cols));
}

// conv1 W[o][i][t] (i < D) -> [pair p][half h][o][8] (tap 2p + h, channel j;
// zero for j >= D; the last pair is a zero tap and the last tap); conv2 W[o][i][t] -> [t][q][o][8]
// with i = 8 q + j; biases as FP32.
template <int D>
__global__ void cls_pack_kernel(const float *__restrict__ w, int64_t off_w1, int64_t off_b1,
                                int64_t off_w2, int64_t off_b2, uint8_t *__restrict__ out) {
    using G = ClsGeo<D, 1>;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    __nv_bfloat16 *w1 = reinterpret_cast<__nv_bfloat16 *>(out + G::kW1);
    for (int e = tid; e < G::Pairs * 2 * 32 * 8; e += nth) {
        const int j = e % 8, o = (e / 8) % 32, h = (e / 256) % 2, p = e / 512;
        // the odd last tap is the second of its step, behind the zero rows
        const int t = p < G::Pairs - 1 ? 2 * p + h : h == 1 ? G::Taps - 1 : -1;
        w1[e] = __float2bfloat16_rn(t >= 0 && j < D ? w[off_w1 + (o * D + j) * G::Taps + t] : 0.f);
    }
    __nv_bfloat16 *w2 = reinterpret_cast<__nv_bfloat16 *>(out + G::kW2);
    for (int e = tid; e < G::Taps * 32 * 32; e += nth) {
        const int t = e / 1024, o = (e / 32) % 32, i = e % 32;
        w2[((t * 4 + i / 8) * 32 + o) * 8 + i % 8] =
            __float2bfloat16_rn(w[off_w2 + (o * 32 + i) * G::Taps + t]);
    }
    for (int i = tid; i < 32; i += nth) {
        reinterpret_cast<float *>(out + G::kB1)[i] = w[off_b1 + i];
        reinterpret_cast<float *>(out + G::kB2)[i] = w[off_b2 + i];
    }
}

template <int D, int NP>
void launch_conv(const DevMesh &m, const float *pool_f, int64_t B, const double *xp,
                 const uint8_t *packed, const FcMat &cat, float *off, int *err, int sm_count,
                 cudaStream_t st) {
    using G = ClsGeo<D, NP>;
    static std::atomic<uint64_t> done{0};
    allow_smem(done, reinterpret_cast<const void *>(cls_conv_tc_kernel<D, NP>), G::kSmTotal);
    const int grid = int(std::min<int64_t>((B + NP - 1) / NP, int64_t(sm_count) * G::PerSm));
    cls_conv_tc_kernel<D, NP><<<grid, G::Threads, G::kSmTotal, st>>>(m, pool_f, B, xp, packed, cat,
                                                                    off, err);
}

}  // namespace

int64_t cls_packed_bytes(int dim) { return dim == 2 ? ClsGeo<2, 1>::kPacked : ClsGeo<3, 1>::kPacked; }

void launch_cls_pack(int dim, const float *w, int64_t off_w1, int64_t off_b1, int64_t off_w2,
                     int64_t off_b2, uint8_t *packed, cudaStream_t st) {
    if (dim == 2)
        cls_pack_kernel<2><<<32, 256, 0, st>>>(w, off_w1, off_b1, off_w2, off_b2, packed);
    else
        cls_pack_kernel<3><<<64, 256, 0, st>>>(w, off_w1, off_b1, off_w2, off_b2, packed);
}

void launch_cls_conv_tc(const DevMesh &m, const float *pool_f, int64_t B, const double *xp,
                        const uint8_t *packed, const FcMat &cat, float *off, int *err,
                        int sm_count, cudaStream_t st) {
    if (B <= 0) return;
    // groups of five once every CTA gets more than one; a particle per CTA pass
    // spreads fewer particles over more CTAs (a forward pass of 2279 particles by
    // ones 83.0 us, of 2281 by fives 79.4 us)
    if (m.dim == 2 && B >= int64_t(15) * sm_count)
        launch_conv<2, 5>(m, pool_f, B, xp, packed, cat, off, err, sm_count, st);
    else if (m.dim == 2)
        launch_conv<2, 1>(m, pool_f, B, xp, packed, cat, off, err, sm_count, st);
    else
        launch_conv<3, 1>(m, pool_f, B, xp, packed, cat, off, err, sm_count, st);
}

}  // namespace cs
