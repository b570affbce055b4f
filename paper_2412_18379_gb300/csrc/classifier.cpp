// The classifier start predictor (Sec. 2.3, Eq. 7-8) as a sequence of
// kernels: pooled-centroid inputs, two zero-padded convolutions, average
// pooling, the offset branch, fusion, logits; the cross-entropy backward,
// Adam on FP32 master parameters, the training loop, the start element of
// the most probable class, and the C ABI entry points of the classifier.
// Inference fuses inputs, convolutions and pooling (classifier_tc.cu); the
// layers run on tiled BF16 operands (fc_tc.cu). A training step takes its 2-D
// convolutions from train_tc.cu, its 3-D ones from im2col and the general GEMM.
// FP32 operands and batches below 16 rows take im2col and that GEMM throughout.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "classifier.h"
#include "cnn.h"
#include "fc_tc.h"
#include "train_tc.h"

namespace cs {

// Parameter offsets of the classifier of one dimension (layer order conv1,
// conv2, xp1, xp2, fuse, logits; W then b of each)
struct ClsShape {
    int dim, W, P, Pq, taps, n_pool, n_cls, ldc;
    int64_t w_off[6], b_off[6], n_params;
    explicit ClsShape(int d) : dim(d) {
        W = cls_window(d);
        P = cls_cells(d);
        Pq = d == 2 ? (W + 2) * (W + 2) : (W + 2) * (W + 2) * (W + 2);
        taps = d == 2 ? 9 : 27;
        n_pool = cls_pooled(d);
        n_cls = P;
        ldc = n_pool + kClsH1;
        const int64_t rows[6] = {kClsCh, kClsCh, kClsH1, kClsH1, kClsH2, n_cls};
        const int64_t cols[6] = {int64_t(d) * taps, int64_t(kClsCh) * taps, d, kClsH1, ldc, kClsH2};
        int64_t o = 0;
        for (int l = 0; l < 6; ++l) {
            w_off[l] = o;
            o += rows[l] * cols[l];
            b_off[l] = o;
            o += rows[l];
        }
        n_params = o;
    }
};

struct Classifier {
    int dim = 0;
    int64_t n = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *loss = nullptr;
    int64_t t = 0;
    // workspace of the layer-by-layer path: the fully connected layers' buffers for
    // cap rows, the unfused module 1's for cap_conv rows, their backward passes' for
    // cap_grad and cap_gconv rows (0 until a path needs them; a tiled step in 3-D
    // takes module 1's alone)
    int64_t cap = 0, cap_conv = 0, cap_grad = 0, cap_gconv = 0;
    std::vector<void *> ws;
    float *a0 = nullptr, *off = nullptr, *col1 = nullptr, *z1 = nullptr, *y1 = nullptr,
          *a1 = nullptr, *col2 = nullptr, *z2 = nullptr, *cat = nullptr, *h1 = nullptr,
          *r1 = nullptr, *h2 = nullptr, *u = nullptr, *ru = nullptr, *H = nullptr;
    float *gH = nullptr, *gu = nullptr, *gcat = nullptr, *gh2 = nullptr, *gh1 = nullptr,
          *gz2 = nullptr;
    int64_t *idx = nullptr;
    float *splitk = nullptr;
    int64_t splitk_n = 0;
    // per-call buffers of cs_track_classifier / cs_classifier_pairs
    double *xp = nullptr;
    int32_t *starts = nullptr;
    int64_t xp_cap = 0;
    // conv1 and conv2 in the fused kernel's layout, refreshed after the
    // parameters change
    uint8_t *packed = nullptr;
    bool packed_dirty = true;
    // the tiled path (fc_tc.h): activations and gradients of the fully
    // connected layers for fc_cap rows (the gradients' where fc_grad), and the
    // packed weights with the tile widths they were packed for
    std::vector<void *> fcws;
    int64_t fc_cap = 0;
    bool fc_grad = false;
    uint8_t *tcat = nullptr, *tr1 = nullptr, *tru = nullptr, *tgH = nullptr, *tgu = nullptr,
            *tgh2 = nullptr, *tgh1 = nullptr;
    float *toff = nullptr, *tH = nullptr, *tgpool = nullptr;
    int *tcount = nullptr;
    int64_t *tidx = nullptr;
    uint8_t *fcpack = nullptr;
    int pack_bn[3] = {0, 0, 0};
    // module 1 of a 2-D training step for tr_cap rows (train_tc.h)
    std::vector<void *> trws;
    int64_t tr_cap = 0;
    float *ta0 = nullptr, *tz2 = nullptr;
    uint16_t *ty1 = nullptr, *tdz2 = nullptr, *tdz1 = nullptr;
    uint8_t *tcpack = nullptr;
    float *parts = nullptr;      // partial sums of a step's gradients
    int64_t parts_cap = 0;
};

}  // namespace cs

using namespace cs;

namespace {

cs_status fail(cs_ctx *ctx, cs_status code, const std::string &msg) {
    if (ctx) ctx->err = msg;
    return code;
}

#define CCHK(call)                                                                       \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess)                                                           \
            return fail(ctx, CS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

cs::Mesh *find_mesh(cs_ctx *ctx, int32_t id) {
    auto it = ctx->meshes.find(id);
    return it == ctx->meshes.end() ? nullptr : it->second;
}

void free_ws(cs_ctx *ctx, Classifier &C) {
    for (void *p : C.ws) dfree(ctx, p);
    C.ws.clear();
    C.a0 = C.off = C.col1 = C.z1 = C.y1 = C.a1 = C.col2 = C.z2 = C.cat = nullptr;
    C.h1 = C.r1 = C.h2 = C.u = C.ru = C.H = nullptr;
    C.gH = C.gu = C.gcat = C.gh2 = C.gh1 = C.gz2 = nullptr;
    C.idx = nullptr;
    C.splitk = nullptr;
    C.splitk_n = 0;
    C.cap = C.cap_conv = C.cap_grad = C.cap_gconv = 0;
}

void free_list(cs_ctx *ctx, std::vector<void *> &v) {
    for (void *p : v) dfree(ctx, p);
    v.clear();
}

void free_fc(cs_ctx *ctx, Classifier &C) {
    free_list(ctx, C.fcws);
    C.tcat = C.tr1 = C.tru = C.tgH = C.tgu = C.tgh2 = C.tgh1 = nullptr;
    C.toff = C.tH = C.tgpool = nullptr;
    C.tcount = nullptr;
    C.tidx = nullptr;
    C.fc_cap = 0;
    C.fc_grad = false;
}

void free_parts(cs_ctx *ctx, Classifier &C) {
    dfree(ctx, C.parts);
    C.parts = nullptr;
    C.parts_cap = 0;
}

void free_tr(cs_ctx *ctx, Classifier &C) {
    free_list(ctx, C.trws);
    C.ta0 = C.tz2 = nullptr;
    C.ty1 = C.tdz2 = C.tdz1 = nullptr;
    C.tcpack = nullptr;
    C.tr_cap = 0;
}

void release(cs_ctx *ctx, Classifier *C) {
    if (!C) return;
    free_ws(ctx, *C);
    free_fc(ctx, *C);
    free_tr(ctx, *C);
    dfree(ctx, C->fcpack);
    dfree(ctx, C->parts);
    for (void *p : {static_cast<void *>(C->w), static_cast<void *>(C->g),
                    static_cast<void *>(C->m), static_cast<void *>(C->v),
                    static_cast<void *>(C->loss), static_cast<void *>(C->xp),
                    static_cast<void *>(C->starts), static_cast<void *>(C->packed)})
        dfree(ctx, p);
    delete C;
}

template <class T>
cs_status ws_alloc(cs_ctx *ctx, Classifier &C, T **p, int64_t count) {
    cs_status rc = dmalloc_n(ctx, p, size_t(std::max<int64_t>(count, 1)));
    if (rc == CS_OK) C.ws.push_back(*p);
    return rc;
}

template <class T>
cs_status list_alloc(cs_ctx *ctx, std::vector<void *> &v, T **p, int64_t count) {
    cs_status rc = dmalloc_n(ctx, p, size_t(std::max<int64_t>(count, 1)));
    if (rc == CS_OK) v.push_back(*p);
    return rc;
}

// Packed weights of the tiled fully connected layers for products of B rows:
// where each lies in Classifier::fcpack and its tile width. Forward W3, W4,
// W5 (xp2, fuse, logits); backward W5^T, the two column ranges of W4^T, W3^T.
struct FcPlan {
    enum { W3, W4, W5, W5T, W4P, W4H, W3T, Count };
    int rows[Count], K[Count], bn[Count];
    int64_t off[Count], bytes;
    FcPlan(const ClsShape &S, int64_t B, int sm) {
        const int r[Count] = {kClsH1, kClsH2, S.n_cls, kClsH2, S.n_pool, kClsH1, kClsH1};
        const int k[Count] = {kClsH1, S.ldc, kClsH2, S.n_cls, kClsH2, kClsH2, kClsH1};
        bytes = 0;
        for (int i = 0; i < Count; ++i) {
            rows[i] = r[i];
            K[i] = k[i];
            bn[i] = fc_bn(B, r[i], sm);
            off[i] = bytes;
            // room for any tile width
            bytes += int64_t(r[i] + 255) / 256 * 256 * fc_kp(k[i]) * 2 + fc_kp(k[i]) * 2 * 256;
        }
    }
};

// buffers of the tiled fully connected layers for `cap` rows, anew
cs_status alloc_fc(cs_ctx *ctx, Classifier &C, int64_t cap, bool g) {
    free_fc(ctx, C);
    const ClsShape S(C.dim);
    auto &v = C.fcws;
    const int np = fc_kp(S.n_cls);
    cs_status rc;
    if ((rc = list_alloc(ctx, v, &C.tcat, fc_bytes(cap, S.ldc))) ||
        (rc = list_alloc(ctx, v, &C.tr1, fc_bytes(cap, kClsH1))) ||
        (rc = list_alloc(ctx, v, &C.tru, fc_bytes(cap, kClsH2))) ||
        (rc = list_alloc(ctx, v, &C.toff, cap * C.dim)) ||
        (rc = list_alloc(ctx, v, &C.tH, cap * S.n_cls)) ||
        (g && ((rc = list_alloc(ctx, v, &C.tgH, fc_bytes(cap, np))) ||
               (rc = list_alloc(ctx, v, &C.tgu, fc_bytes(cap, kClsH2))) ||
               (rc = list_alloc(ctx, v, &C.tgh2, fc_bytes(cap, kClsH1))) ||
               (rc = list_alloc(ctx, v, &C.tgh1, fc_bytes(cap, kClsH1))) ||
               (rc = list_alloc(ctx, v, &C.tgpool, cap * S.n_pool)) ||
               (rc = list_alloc(ctx, v, &C.tidx, cap)) || (rc = list_alloc(ctx, v, &C.tcount, 1))))) {
        free_fc(ctx, C);
        return rc;
    }
    C.fc_cap = cap;
    C.fc_grad = g;
    return CS_OK;
}

cs_status ensure_fc(cs_ctx *ctx, Classifier &C, int64_t B, bool grad) {
    cs_status rc = ensure_err(ctx);
    if (rc) return rc;
    use_workspace(C.dim, kUseFc);
    const ClsShape S(C.dim);
    if (!C.fcpack) {
        if ((rc = dmalloc_n(ctx, &C.fcpack, size_t(FcPlan(S, 1, ctx->sm_count).bytes)))) return rc;
        C.pack_bn[0] = 0;
    }
    if (C.fc_cap >= B && (!grad || C.fc_grad)) return CS_OK;
    return alloc_fc(ctx, C, std::max(B, C.fc_cap), grad || C.fc_grad);
}

// buffers of module 1 of a 2-D training step
cs_status ensure_tr(cs_ctx *ctx, Classifier &C, int64_t B) {
    use_workspace(C.dim, kUseTrain);
    if (C.tr_cap >= B) return CS_OK;
    free_tr(ctx, C);
    const ClsShape S(2);
    auto &v = C.trws;
    cs_status rc;
    if ((rc = list_alloc(ctx, v, &C.ta0, B * 2 * S.Pq)) ||
        (rc = list_alloc(ctx, v, &C.tz2, B * S.P * kClsCh)) ||
        (rc = list_alloc(ctx, v, &C.ty1, B * S.Pq * kClsCh)) ||
        (rc = list_alloc(ctx, v, &C.tdz2, B * S.P * kClsCh)) ||
        (rc = list_alloc(ctx, v, &C.tdz1, B * S.P * kClsCh)) ||
        (rc = list_alloc(ctx, v, &C.tcpack, 64 * 1024))) {
        free_tr(ctx, C);
        return rc;
    }
    // the zero ring of conv2's input: only the interior is ever written
    if (cudaMemset(C.ty1, 0, size_t(B) * S.Pq * kClsCh * 2) != cudaSuccess) {
        free_tr(ctx, C);
        return fail(ctx, CS_ECUDA, "cudaMemset of the padded activations failed");
    }
    C.tr_cap = B;
    return CS_OK;
}

// Workspace of the layer-by-layer path for B rows of the named parts: the fully
// connected layers, module 1 (with the GEMMs' K splits; no product of the layers
// alone splits its K off the tensor cores), and their backward passes (module 1's
// reuses its forward buffers). Growing any part reallocates all of them, each at
// its own row count.
enum : unsigned { kWsFc = 1, kWsConv = 2, kWsFcGrad = 4, kWsConvGrad = 8 };
constexpr unsigned kWsAll = kWsFc | kWsConv | kWsFcGrad | kWsConvGrad;

// K splits of module 1's products alone: at most three of a forward product of
// less than two waves of tiles, 128 x 32 floats each (the weight gradients', of at
// most 32 x 864, take less)
int64_t conv_splitk_floats(int sm_count) { return int64_t(3) * 2 * sm_count * 128 * kClsCh; }

// the parts at rows[0..3] and a K-split workspace of sk floats, all anew
cs_status alloc_ws(cs_ctx *ctx, Classifier &C, const int64_t (&rows)[4], int64_t sk) {
    free_ws(ctx, C);
    const ClsShape S(C.dim);
    const int64_t d = C.dim, K1 = d * S.taps, K2 = int64_t(kClsCh) * S.taps;
    const int64_t r = rows[0], rv = rows[1], rg = rows[2], rgv = rows[3];
    cs_status rc = CS_OK;
    if ((r > 0 && ((rc = ws_alloc(ctx, C, &C.off, r * d)) || (rc = ws_alloc(ctx, C, &C.cat, r * S.ldc)) ||
                   (rc = ws_alloc(ctx, C, &C.h1, r * kClsH1)) ||
                   (rc = ws_alloc(ctx, C, &C.r1, r * kClsH1)) ||
                   (rc = ws_alloc(ctx, C, &C.h2, r * kClsH1)) ||
                   (rc = ws_alloc(ctx, C, &C.u, r * kClsH2)) ||
                   (rc = ws_alloc(ctx, C, &C.ru, r * kClsH2)) ||
                   (rc = ws_alloc(ctx, C, &C.H, r * S.n_cls)))) ||
        (sk > 0 && (rc = ws_alloc(ctx, C, &C.splitk, sk))) ||
        (rv > 0 && ((rc = ws_alloc(ctx, C, &C.a0, rv * d * S.Pq)) ||
                    (rc = ws_alloc(ctx, C, &C.col1, rv * S.P * K1)) ||
                    (rc = ws_alloc(ctx, C, &C.z1, rv * S.P * kClsCh)) ||
                    (rc = ws_alloc(ctx, C, &C.y1, rv * S.P * kClsCh)) ||
                    (rc = ws_alloc(ctx, C, &C.a1, rv * S.Pq * kClsCh)) ||
                    (rc = ws_alloc(ctx, C, &C.col2, rv * S.P * K2)) ||
                    (rc = ws_alloc(ctx, C, &C.z2, rv * S.P * kClsCh)))) ||
        (rg > 0 && ((rc = ws_alloc(ctx, C, &C.gH, rg * S.n_cls)) ||
                    (rc = ws_alloc(ctx, C, &C.gu, rg * kClsH2)) ||
                    (rc = ws_alloc(ctx, C, &C.gcat, rg * S.ldc)) ||
                    (rc = ws_alloc(ctx, C, &C.gh2, rg * kClsH1)) ||
                    (rc = ws_alloc(ctx, C, &C.gh1, rg * kClsH1)) || (rc = ws_alloc(ctx, C, &C.idx, rg)))) ||
        (rgv > 0 && (rc = ws_alloc(ctx, C, &C.gz2, rgv * S.P * kClsCh)))) {
        free_ws(ctx, C);
        return rc;
    }
    C.splitk_n = sk;
    C.cap = r;
    C.cap_conv = rv;
    C.cap_grad = rg;
    C.cap_gconv = rgv;
    return CS_OK;
}

cs_status ensure_ws(cs_ctx *ctx, Classifier &C, int64_t B, unsigned what) {
    cs_status rc = ensure_err(ctx);
    if (rc) return rc;
    use_workspace(C.dim, kUseWs);
    const int64_t caps[4] = {C.cap, C.cap_conv, C.cap_grad, C.cap_gconv};
    int64_t rows[4];
    bool fits = true;
    for (int i = 0; i < 4; ++i) {
        rows[i] = (what >> i) & 1u ? std::max(B, caps[i]) : caps[i];
        fits = fits && rows[i] == caps[i];
    }
    const int64_t sk = !(what & kWsConv) ? 0
                       : what & kWsFc    ? tc_gemm_work_floats(ctx->sm_count)
                                         : conv_splitk_floats(ctx->sm_count);
    if (fits && C.splitk_n >= sk) return CS_OK;
    return alloc_ws(ctx, C, rows, std::max(sk, C.splitk_n));
}

// need(): the workspaces of a call. Where memory has no room for them beside what
// calls before left in the same sets (rows, gradients), they are made anew; a call
// that is refused leaves none.
template <class F>
cs_status with_room(cs_ctx *ctx, Classifier &C, F need) {
    const std::string message = ctx->err;
    cs_status rc = need();
    for (int i = 0; i < 2 && rc == CS_ENOMEM; ++i) {
        free_ws(ctx, C);
        free_fc(ctx, C);
        free_tr(ctx, C);
        free_parts(ctx, C);
        if (i == 0 && (rc = need()) == CS_OK) ctx->err = message;
    }
    return rc;
}

int gemm(cs_ctx *ctx, Classifier &C, const float *A, const float *Bm, float *Cm, const float *bias,
         int64_t M, int64_t N, int64_t K, bool transA, bool transB, cudaStream_t st) {
    return launch_gemm(A, Bm, Cm, bias, M, N, K, transA, transB, false, st, ctx->dev_err,
                       ctx->sm_count, C.splitk, C.splitk_n);
}

int relu(cs_ctx *ctx, const float *z, float *y, int64_t n, cudaStream_t st) {
    return launch_relu(z, y, n, ctx->sm_count, st);
}

// module 2, fusion and logits of B rows whose pooled features (C.cat's
// first n_pool columns) and offsets (C.off) are in place, into C.H
int forward_fc(cs_ctx *ctx, Classifier &C, int64_t B, cudaStream_t st) {
    const ClsShape S(C.dim);
    const int sm = ctx->sm_count, d = C.dim;
    int n = 0;
    // module 2: the offset of x_p through two fully connected layers
    n += gemm(ctx, C, C.off, C.w + S.w_off[2], C.h1, C.w + S.b_off[2], B, kClsH1, d, false, true,
              st);
    n += relu(ctx, C.h1, C.r1, B * kClsH1, st);
    n += gemm(ctx, C, C.r1, C.w + S.w_off[3], C.h2, C.w + S.b_off[3], B, kClsH1, kClsH1, false,
              true, st);
    launch_cls_cat_relu(C.h2, B, kClsH1, C.cat, S.ldc, S.n_pool, sm, st);
    n += 1;
    // fusion and logits
    n += gemm(ctx, C, C.cat, C.w + S.w_off[4], C.u, C.w + S.b_off[4], B, kClsH2, S.ldc, false,
              true, st);
    n += relu(ctx, C.u, C.ru, B * kClsH2, st);
    n += gemm(ctx, C, C.ru, C.w + S.w_off[5], C.H, C.w + S.b_off[5], B, S.n_cls, kClsH2, false,
              true, st);
    return n;
}

// ---------------------------------------------------------------------------
// The tiled path: BF16 operands (fc_tc.h, train_tc.h)
// ---------------------------------------------------------------------------

// refresh the packed weights of the fully connected layers
int pack_fc(cs_ctx *ctx, Classifier &C, const ClsShape &S, const FcPlan &P, bool grad,
            cudaStream_t st) {
    const float *w = C.w;
    const float *W3 = w + S.w_off[3], *W4 = w + S.w_off[4], *W5 = w + S.w_off[5];
    auto seg = [&](int i, const float *W, int64_t rs, int64_t ks) {
        return FcPack{W, rs, ks, P.rows[i], P.K[i], P.bn[i], C.fcpack + P.off[i]};
    };
    FcPack f[FcPlan::Count] = {seg(FcPlan::W3, W3, kClsH1, 1), seg(FcPlan::W4, W4, S.ldc, 1),
                               seg(FcPlan::W5, W5, kClsH2, 1), seg(FcPlan::W5T, W5, 1, kClsH2),
                               seg(FcPlan::W4P, W4, 1, S.ldc), seg(FcPlan::W4H, W4 + S.n_pool, 1, S.ldc),
                               seg(FcPlan::W3T, W3, 1, kClsH1)};
    return launch_fc_pack(f, grad ? int(FcPlan::Count) : 3, st);
}

// module 2, fusion and logits of B rows whose pooled features (C.tcat's first
// columns) and offsets (C.toff) are in place, into H
int fc_forward(cs_ctx *ctx, Classifier &C, const ClsShape &S, const FcPlan &P, int64_t B, float *H,
               cudaStream_t st) {
    const int sm = ctx->sm_count;
    const FcMat cat = fc_mat(C.tcat, S.ldc), r1 = fc_mat(C.tr1, kClsH1), ru = fc_mat(C.tru, kClsH2);
    int n = launch_fc_offset(C.dim, B, C.toff, C.w + S.w_off[2], C.w + S.b_off[2], r1, sm, st);
    FcGemm g{r1, C.fcpack + P.off[FcPlan::W3], P.bn[FcPlan::W3], kClsH1, B};
    g.bias = C.w + S.b_off[3];
    g.relu = true;
    g.out = fc_cols(cat, S.n_pool, kClsH1);
    n += launch_fc_gemm(g, ctx->dev_err, sm, st);
    FcGemm u{cat, C.fcpack + P.off[FcPlan::W4], P.bn[FcPlan::W4], kClsH2, B};
    u.bias = C.w + S.b_off[4];
    u.relu = true;
    u.out = ru;
    fc_split_like_gemm(B, kClsH2, S.ldc, sm, &u.nsplit, &u.kc);
    n += launch_fc_gemm(u, ctx->dev_err, sm, st);
    FcGemm l{ru, C.fcpack + P.off[FcPlan::W5], P.bn[FcPlan::W5], S.n_cls, B};
    l.bias = C.w + S.b_off[5];
    l.f32 = H;
    l.ldf = S.n_cls;
    return n + launch_fc_gemm(l, ctx->dev_err, sm, st);
}

// Batches that the tiled path takes: BF16 operands and at least 16 rows. Below
// 16 the GEMM's products do not run on the tensor cores, and their sums round
// differently; such a batch or chunk keeps those layers, so that its results do
// not depend on which kernels the larger ones use. (A gradient call of 15 rows
// takes 576 us in 2-D and 720 in 3-D, one of 16 206 and 423.)
bool tiled_batch(int64_t B) { return gemm_bf16() && B >= 16; }

// inference of B particles xp[b] into H [B][n_cls]: module 1 fused on the
// tensor cores, then the tiled fully connected layers or, for less than a tiled
// batch, those of the training path (its BF16 features widened to FP32 lose
// nothing: that path rounds its operands to BF16 itself)
int infer(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t B, const double *xp, float *H,
          cudaStream_t st) {
    const ClsShape S(C.dim);
    const FcPlan P(S, B, ctx->sm_count);
    int n = 0;
    if (C.packed_dirty) {
        launch_cls_pack(C.dim, C.w, S.w_off[0], S.b_off[0], S.w_off[1], S.b_off[1], C.packed, st);
        n += 1;
    }
    const bool tiled = tiled_batch(B);
    if (C.packed_dirty) C.pack_bn[0] = 0;
    if (tiled && !std::equal(C.pack_bn, C.pack_bn + 3, P.bn)) {
        n += pack_fc(ctx, C, S, P, false, st);
        std::copy(P.bn, P.bn + 3, C.pack_bn);
    }
    C.packed_dirty = false;
    const FcMat cat = fc_mat(C.tcat, S.ldc);
    launch_cls_conv_tc(m, m.pool_f, B, xp, C.packed, cat, tiled ? C.toff : C.off, ctx->dev_err,
                       ctx->sm_count, st);
    n += 1;
    if (tiled) return n + fc_forward(ctx, C, S, P, B, H, st);
    n += launch_fc_widen(fc_cols(cat, 0, S.n_pool), B, C.cat, S.ldc, st);
    n += forward_fc(ctx, C, B, st);
    if (H != C.H)
        cudaMemcpyAsync(H, C.H, size_t(B) * S.n_cls * sizeof(float), cudaMemcpyDeviceToDevice, st);
    return n;
}

int forward_conv(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t B, const double *xp,
                 const int64_t *idx, float *off, cudaStream_t st);
int backward_conv(cs_ctx *ctx, Classifier &C, int64_t B, const float *dpool, int64_t ld,
                  cudaStream_t st);

// The tiled path's training step for B rows (tiled_batch): gradients of the
// cross-entropy into C.g, and *loss. In 2-D module 1 runs on the
// implicit-GEMM convolutions as well (train_tc.h); in 3-D, whose 343 positions
// do not fit their tile, on the layer-by-layer kernels.

// floats of a step's partial sums
int64_t train_parts(cs_ctx *ctx, const ClsShape &S, int64_t B) {
    const int sm = ctx->sm_count;
    const int64_t mt = (B + 127) / 128;
    int64_t n = int64_t(fc_wgrad_splits(B, S.n_cls, kClsH2, sm)) * S.n_cls * kClsH2 +
                int64_t(fc_wgrad_splits(B, kClsH2, S.ldc, sm)) * kClsH2 * S.ldc +
                int64_t(fc_wgrad_splits(B, kClsH1, kClsH1, sm)) * kClsH1 * kClsH1;
    n += cls_softmax_blocks(B) * (int64_t(S.n_cls) + 1);
    n += 4 * mt * (kClsH2 + 2 * kClsH1) + mt * kClsH1 * S.dim;
    if (S.dim == 2)
        n += 2 * int64_t(sm) * kClsCh * (kClsCh * S.taps + 2 * S.taps + 1) +
             int64_t(cls_pool_back_blocks(B, sm)) * kClsCh;
    return n;
}

cs_status ensure_train(cs_ctx *ctx, Classifier &C, int64_t B) {
    cs_status rc = ensure_fc(ctx, C, B, true);
    if (rc == CS_OK) rc = C.dim == 2 ? ensure_tr(ctx, C, B) : ensure_ws(ctx, C, B, kWsConv | kWsConvGrad);
    if (rc) return rc;
    use_workspace(C.dim, kUseParts);
    const int64_t need = train_parts(ctx, ClsShape(C.dim), B);
    if (C.parts_cap >= need) return CS_OK;
    free_parts(ctx, C);
    if ((rc = dmalloc_n(ctx, &C.parts, size_t(need)))) return rc;
    C.parts_cap = need;
    return CS_OK;
}

int train_tiled(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t B, const double *xp,
                const int32_t *labels, const int64_t *idx, float *loss, cudaStream_t st) {
    const ClsShape S(C.dim);
    const FcPlan P(S, B, ctx->sm_count);
    const int sm = ctx->sm_count, d = C.dim;
    int *err = ctx->dev_err;
    float *g = C.g;
    int n = pack_fc(ctx, C, S, P, true, st);
    C.pack_bn[0] = 0;            // inference packs its own widths again
    const FcMat cat = fc_mat(C.tcat, S.ldc), r1 = fc_mat(C.tr1, kClsH1), ru = fc_mat(C.tru, kClsH2);
    const FcMat gH = fc_mat(C.tgH, fc_kp(S.n_cls)), gu = fc_mat(C.tgu, kClsH2);
    const FcMat gh2 = fc_mat(C.tgh2, kClsH1), gh1 = fc_mat(C.tgh1, kClsH1);
    const ConvGeo c1(2, 2, 11), c2(2, kClsCh, 11);
    // 2 KB, 18 KB and 18 KB
    uint8_t *f1 = C.tcpack, *f2 = f1 + 4 * 1024, *b2 = f2 + 20 * 1024;
    if (d == 2) {
        const PackSeg ps[2] = {{C.w + S.w_off[0], c1.K, 0, f1, nullptr, nullptr},
                               {C.w + S.w_off[1], c2.K, train_packed_kw(2), f2, b2, nullptr}};
        n += launch_pack_train(ps, 2, st);
        launch_cls_features(m, B, xp, idx, true, C.ta0, C.toff, sm, st);
        n += 1 + launch_conv_fwd(c1, C.ta0, true, B, f1, C.w + S.b_off[0], C.ty1, 1, nullptr, err, sm, st);
        n += launch_conv_fwd(c2, C.ty1, false, B, f2, C.w + S.b_off[1], nullptr, 0, C.tz2, err, sm, st);
    } else {
        n += forward_conv(ctx, C, m, B, xp, idx, C.toff, st);
    }
    const float *z2 = d == 2 ? C.tz2 : C.z2;
    launch_cls_pool_tiled(d, z2, B, cat, sm, st);
    n += 1 + fc_forward(ctx, C, S, P, B, C.tH, st);

    ReduceSeg seg[kMaxSegs];
    int ns = 0;
    float *part = C.parts;
    auto sum = [&](int64_t count, int parts, float *out) {
        float *p = part;
        seg[ns++] = ReduceSeg{p, count, count, out, parts, 0.f};
        part += count * parts;
        return p;
    };
    auto wgrad = [&](const FcMat &Y, const FcMat &X, int N, int K, int64_t w_off) {
        const int s = fc_wgrad_splits(B, N, K, sm);
        n += launch_fc_wgrad(Y, X, B, N, K, s, sum(int64_t(N) * K, s, g + w_off), err, st);
    };
    const int mt = int((B + 127) / 128), sb = cls_softmax_blocks(B);
    // logits
    float *b5 = sum(S.n_cls, sb, g + S.b_off[5]);
    float *lp = part;
    part += sb;
    launch_softmax_ce_tiled(C.tH, labels, idx, B, S.n_cls, gH, b5, lp, C.tcount, st);
    launch_loss_sum(lp, sb, C.tcount, loss, st);
    n += 3;
    wgrad(gH, ru, S.n_cls, kClsH2, S.w_off[5]);
    // fusion
    FcGemm q{gH, C.fcpack + P.off[FcPlan::W5T], P.bn[FcPlan::W5T], kClsH2, B};
    q.gate = ru;
    q.out = gu;
    q.colsum = sum(kClsH2, 4 * mt, g + S.b_off[4]);
    n += launch_fc_gemm(q, err, sm, st);
    wgrad(gu, cat, kClsH2, S.ldc, S.w_off[4]);
    FcGemm gp{gu, C.fcpack + P.off[FcPlan::W4P], P.bn[FcPlan::W4P], S.n_pool, B};
    gp.f32 = C.tgpool;
    gp.ldf = S.n_pool;
    n += launch_fc_gemm(gp, err, sm, st);
    // module 2
    FcGemm q2{gu, C.fcpack + P.off[FcPlan::W4H], P.bn[FcPlan::W4H], kClsH1, B};
    q2.gate = fc_cols(cat, S.n_pool, kClsH1);
    q2.out = gh2;
    q2.colsum = sum(kClsH1, 4 * mt, g + S.b_off[3]);
    n += launch_fc_gemm(q2, err, sm, st);
    wgrad(gh2, r1, kClsH1, kClsH1, S.w_off[3]);
    FcGemm q1{gh2, C.fcpack + P.off[FcPlan::W3T], P.bn[FcPlan::W3T], kClsH1, B};
    q1.gate = r1;
    q1.out = gh1;
    q1.colsum = sum(kClsH1, 4 * mt, g + S.b_off[2]);
    n += launch_fc_gemm(q1, err, sm, st);
    n += launch_fc_offset_grad(d, B, C.toff, gh1, sum(int64_t(kClsH1) * d, mt, g + S.w_off[2]), st);
    // module 1
    if (d == 2) {
        const int pb = cls_pool_back_blocks(B, sm);
        launch_cls_pool_back_tiled(C.tgpool, z2, B, C.tdz2, sum(kClsCh, pb, g + S.b_off[1]), sm, st);
        const int ca2 = conv_bwd_ctas(c2, B, false, sm), ca1 = conv_bwd_ctas(c1, B, true, sm);
        float *w2 = sum(int64_t(kClsCh) * c2.K, ca2, g + S.w_off[1]);
        float *bb1 = sum(kClsCh, ca2, g + S.b_off[0]);
        n += 1 + launch_conv_bwd(c2, C.ty1, false, B, C.tdz2, b2, w2, C.tdz1, bb1, err, sm, st);
        float *w1 = sum(int64_t(kClsCh) * c1.K, ca1, g + S.w_off[0]);
        n += launch_conv_bwd(c1, C.ta0, true, B, C.tdz1, nullptr, w1, nullptr, nullptr, err, sm, st);
    } else {
        n += backward_conv(ctx, C, B, C.tgpool, S.n_pool, st);
    }
    return n + launch_reduce_parts(seg, ns, st);
}

// forward of B rows (particles xp[idx[b]], or xp[b]) into C.H [B][n_cls],
// keeping every activation the backward pass reads
int forward(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t B, const double *xp,
            const int64_t *idx, cudaStream_t st) {
    const ClsShape S(C.dim);
    const int n = forward_conv(ctx, C, m, B, xp, idx, C.off, st);
    launch_cls_pool(C.dim, C.z2, B, C.cat, S.ldc, ctx->sm_count, st);
    return n + 1 + forward_fc(ctx, C, B, st);
}

// module 1 of B rows into C.z2 (before its ReLU), the offsets into `off`
int forward_conv(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t B, const double *xp,
                 const int64_t *idx, float *off, cudaStream_t st) {
    const ClsShape S(C.dim);
    const int sm = ctx->sm_count, d = C.dim;
    const int64_t BP = B * S.P;
    int n = 0;
    launch_cls_features(m, B, xp, idx, true, C.a0, off, sm, st);
    n += 1;
    // module 1: two zero-padded 3^d convolutions with ReLU, pooling
    n += launch_im2col(d, C.a0, B, d, S.W + 2, true, C.col1, sm, st);
    n += gemm(ctx, C, C.col1, C.w + S.w_off[0], C.z1, C.w + S.b_off[0], BP, kClsCh,
              int64_t(d) * S.taps, false, true, st);
    n += relu(ctx, C.z1, C.y1, BP * kClsCh, st);
    launch_cls_pad(d, C.y1, B, kClsCh, C.a1, sm, st);
    n += 1;
    n += launch_im2col(d, C.a1, B, kClsCh, S.W + 2, false, C.col2, sm, st);
    n += gemm(ctx, C, C.col2, C.w + S.w_off[1], C.z2, C.w + S.b_off[1], BP, kClsCh,
              int64_t(kClsCh) * S.taps, false, true, st);
    return n;
}

// gradients of the cross-entropy of C.H against labels[idx[b]] into C.g;
// the loss is added to *loss. Buffers no longer needed are reused: col2
// takes the gradient of its columns, a1 that of the padded input, y1 that of
// the first convolution's output.
int backward(cs_ctx *ctx, Classifier &C, int64_t B, const int32_t *labels, const int64_t *idx,
             float *loss, cudaStream_t st) {
    const ClsShape S(C.dim);
    const int sm = ctx->sm_count, d = C.dim;
    float *g = C.g;
    const float *w = C.w;
    int n = 0;
    launch_softmax_ce(C.H, labels, idx, B, S.n_cls, C.gH, loss, st);
    n += 1;
    // logits and fusion
    n += gemm(ctx, C, C.gH, C.ru, g + S.w_off[5], nullptr, S.n_cls, kClsH2, B, true, false, st);
    n += launch_colsum(C.gH, B, S.n_cls, g + S.b_off[5], st, C.splitk, C.splitk_n, sm);
    n += gemm(ctx, C, C.gH, w + S.w_off[5], C.gu, nullptr, B, kClsH2, S.n_cls, false, false, st);
    n += launch_relu_back(C.u, C.gu, B * kClsH2, sm, st);
    n += gemm(ctx, C, C.gu, C.cat, g + S.w_off[4], nullptr, kClsH2, S.ldc, B, true, false, st);
    n += launch_colsum(C.gu, B, kClsH2, g + S.b_off[4], st, C.splitk, C.splitk_n, sm);
    n += gemm(ctx, C, C.gu, w + S.w_off[4], C.gcat, nullptr, B, S.ldc, kClsH2, false, false, st);
    // module 2
    launch_cls_uncat_relu_back(C.gcat, S.ldc, S.n_pool, C.h2, B, kClsH1, C.gh2, sm, st);
    n += 1;
    n += gemm(ctx, C, C.gh2, C.r1, g + S.w_off[3], nullptr, kClsH1, kClsH1, B, true, false, st);
    n += launch_colsum(C.gh2, B, kClsH1, g + S.b_off[3], st, C.splitk, C.splitk_n, sm);
    n += gemm(ctx, C, C.gh2, w + S.w_off[3], C.gh1, nullptr, B, kClsH1, kClsH1, false, false, st);
    n += launch_relu_back(C.h1, C.gh1, B * kClsH1, sm, st);
    n += gemm(ctx, C, C.gh1, C.off, g + S.w_off[2], nullptr, kClsH1, d, B, true, false, st);
    n += launch_colsum(C.gh1, B, kClsH1, g + S.b_off[2], st, C.splitk, C.splitk_n, sm);
    return n + backward_conv(ctx, C, B, C.gcat, S.ldc, st);
}

// module 1's gradients from that of the pooled features (dpool, row stride
// ld): pooling, second and first convolution
int backward_conv(cs_ctx *ctx, Classifier &C, int64_t B, const float *dpool, int64_t ld,
                  cudaStream_t st) {
    const ClsShape S(C.dim);
    const int sm = ctx->sm_count, d = C.dim;
    const int64_t BP = B * S.P;
    float *g = C.g;
    const float *w = C.w;
    int n = 0;
    launch_cls_pool_back(d, dpool, ld, C.z2, B, C.gz2, sm, st);
    n += 1;
    const int64_t K2 = int64_t(kClsCh) * S.taps;
    n += gemm(ctx, C, C.gz2, C.col2, g + S.w_off[1], nullptr, kClsCh, K2, BP, true, false, st);
    n += launch_colsum(C.gz2, BP, kClsCh, g + S.b_off[1], st, C.splitk, C.splitk_n, sm);
    float *dcol2 = C.col2, *dpad = C.a1, *gz1 = C.y1;
    n += gemm(ctx, C, C.gz2, w + S.w_off[1], dcol2, nullptr, BP, K2, kClsCh, false, false, st);
    n += launch_col2im(d, dcol2, B, kClsCh, S.W + 2, dpad, sm, st);
    launch_cls_crop_relu_back(d, dpad, C.z1, B, kClsCh, gz1, sm, st);
    n += 1;
    n += gemm(ctx, C, gz1, C.col1, g + S.w_off[0], nullptr, kClsCh, int64_t(d) * S.taps, BP, true,
              false, st);
    n += launch_colsum(gz1, BP, kClsCh, g + S.b_off[0], st, C.splitk, C.splitk_n, sm);
    return n;
}

Classifier *get_cls(cs_ctx *ctx, int dim) {
    if (dim != 2 && dim != 3) return nullptr;
    return ctx->cls[dim - 2];
}

uint64_t splitmix(uint64_t &s) {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// rows per forward chunk. The fused path needs only the fully connected
// layers' buffers (about 3.4 KB a row in 2-D, 5.2 KB in 3-D): chunks of this
// size give those products enough tiles to fill the GPU without splitting K.
// The unfused path's im2col buffers take about 1 GB at its smaller chunks.
int64_t chunk_rows(int dim, bool fused) {
    if (fused) return dim == 2 ? 32768 : 16384;
    return dim == 2 ? 8192 : 1024;
}

cs_status ensure_xp(cs_ctx *ctx, Classifier &C, int64_t n) {
    if (C.xp_cap >= n) return CS_OK;
    dfree(ctx, C.xp);
    dfree(ctx, C.starts);
    C.xp = nullptr;
    C.starts = nullptr;
    C.xp_cap = 0;
    cs_status rc;
    if ((rc = dmalloc_n(ctx, &C.xp, size_t(n) * C.dim)) ||
        (rc = dmalloc_n(ctx, &C.starts, size_t(n))))
        return rc;
    C.xp_cap = n;
    return CS_OK;
}

// logits of n particles, chunk by chunk, into dst [n][n_cls] or, without it,
// into a chunk's own buffer, which `each` reads before the next chunk
template <class F>
cs_status forward_chunks(cs_ctx *ctx, Classifier &C, const DevMesh &m, int64_t n, const double *xp,
                         float *dst, cudaStream_t st, F each) {
    const bool fused = gemm_bf16();
    WorkspaceScope use;
    const int ncls = cls_cells(C.dim);
    const int64_t R = std::min<int64_t>(n, chunk_rows(C.dim, fused));
    // a chunk, the last one, of less than a tiled batch
    const int64_t rest = n % R > 0 ? n % R : R;
    cs_status rc = with_room(ctx, C, [&] {
        if (!fused) return ensure_ws(ctx, C, R, kWsFc | kWsConv);
        const cs_status r = ensure_fc(ctx, C, R, false);
        return r == CS_OK && !tiled_batch(rest) ? ensure_ws(ctx, C, rest, kWsFc) : r;
    });
    if (rc) return rc;
    for (int64_t r0 = 0; r0 < n; r0 += R) {
        const int64_t B = std::min(R, n - r0);
        float *H = dst ? dst + r0 * ncls : fused && tiled_batch(B) ? C.tH : C.H;
        if (fused) {
            ctx->launches += infer(ctx, C, m, B, xp + r0 * C.dim, H, st);
        } else {
            ctx->launches += forward(ctx, C, m, B, xp + r0 * C.dim, nullptr, st);
            if (dst && cudaMemcpyAsync(H, C.H, size_t(B) * ncls * sizeof(float),
                                       cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                return fail(ctx, CS_ECUDA, "copy of the logits failed");
        }
        if ((rc = each(r0, B, H))) return rc;
    }
    return CS_OK;
}

}  // namespace

namespace cs {
bool classifier_reclaim(cs_ctx *ctx) {
    bool any = false;
    for (Classifier *C : ctx->cls) {
        if (!C) continue;
        if (!in_use(C->dim, kUseWs) && !C->ws.empty()) {
            free_ws(ctx, *C);
            any = true;
        }
        if (!in_use(C->dim, kUseFc) && C->fcpack) {
            free_fc(ctx, *C);
            dfree(ctx, C->fcpack);
            C->fcpack = nullptr;
            any = true;
        }
        if (!in_use(C->dim, kUseTrain) && !C->trws.empty()) {
            free_tr(ctx, *C);
            any = true;
        }
        if (!in_use(C->dim, kUseParts) && C->parts) {
            free_parts(ctx, *C);
            any = true;
        }
    }
    return any;
}

void classifier_release_all(cs_ctx *ctx) {
    for (auto &c : ctx->cls) {
        release(ctx, c);
        c = nullptr;
    }
}
}  // namespace cs

extern "C" {

int64_t cs_classifier_size(int dim) {
    if (dim != 2 && dim != 3) return 0;
    return ClsShape(dim).n_params;
}

int32_t cs_classifier_window(int dim) {
    if (dim != 2 && dim != 3) return 0;
    return cls_window(dim);
}

cs_status cs_classifier_load(cs_ctx *ctx, int dim, const float *params, int64_t n) {
    if (!ctx) return CS_EINVAL;
    if ((dim != 2 && dim != 3) || !params || n != cs_classifier_size(dim))
        return fail(ctx, CS_EINVAL, "cs_classifier_load: bad dim or size (expected " +
                                        std::to_string(cs_classifier_size(dim)) + " floats)");
    if (ctx->server) return fail(ctx, CS_EBUSY, "cs_classifier_load: stop serving first");
    CCHK(cudaSetDevice(ctx->device));
    CCHK(cudaDeviceSynchronize());
    release(ctx, ctx->cls[dim - 2]);
    ctx->cls[dim - 2] = nullptr;
    Classifier *C = new (std::nothrow) Classifier();
    if (!C) return fail(ctx, CS_ENOMEM, "host allocation failed");
    C->dim = dim;
    C->n = n;
    cs_status rc;
    if ((rc = dmalloc_n(ctx, &C->w, size_t(n))) || (rc = dmalloc_n(ctx, &C->g, size_t(n))) ||
        (rc = dmalloc_n(ctx, &C->m, size_t(n))) || (rc = dmalloc_n(ctx, &C->v, size_t(n))) ||
        (rc = dmalloc_n(ctx, &C->loss, 1)) ||
        (rc = dmalloc_n(ctx, &C->packed, size_t(cls_packed_bytes(dim))))) {
        release(ctx, C);
        return rc;
    }
    if (cudaMemcpy(C->w, params, size_t(n) * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(C->m, 0, size_t(n) * sizeof(float)) != cudaSuccess ||
        cudaMemset(C->v, 0, size_t(n) * sizeof(float)) != cudaSuccess) {
        release(ctx, C);
        return fail(ctx, CS_ECUDA, "cs_classifier_load: copy of the parameters failed");
    }
    ctx->cls[dim - 2] = C;
    return CS_OK;
}

cs_status cs_classifier_save(cs_ctx *ctx, int dim, float *out, int64_t n) {
    if (!ctx) return CS_EINVAL;
    if ((dim != 2 && dim != 3) || !out || n != cs_classifier_size(dim))
        return fail(ctx, CS_EINVAL, "cs_classifier_save: bad dim or size");
    Classifier *C = get_cls(ctx, dim);
    if (!C) return fail(ctx, CS_ENOPRED, "cs_classifier_save: no classifier loaded");
    CCHK(cudaSetDevice(ctx->device));
    CCHK(cudaDeviceSynchronize());
    CCHK(cudaMemcpy(out, C->w, size_t(n) * sizeof(float), cudaMemcpyDeviceToHost));
    return CS_OK;
}

cs_status cs_departure(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *x, const double *u,
                       double dt, double *xp_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_departure: unknown mesh id");
    if (n < 0 || (n > 0 && (!x || !u || !xp_out)))
        return fail(ctx, CS_EINVAL, "cs_departure: bad arguments");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    launch_departure(n, m->d.dim, x, u, dt, xp_out, ctx->sm_count,
                     static_cast<cudaStream_t>(stream));
    ctx->launches += 1;
    CCHK(cudaGetLastError());
    return CS_OK;
}

cs_status cs_classifier_features(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *xp,
                                 float *window_out, float *offset_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_features: unknown mesh id");
    if (n < 0 || (n > 0 && (!xp || !window_out || !offset_out)))
        return fail(ctx, CS_EINVAL, "cs_classifier_features: bad arguments");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    launch_cls_features(m->d, n, xp, nullptr, false, window_out, offset_out, ctx->sm_count,
                        static_cast<cudaStream_t>(stream));
    ctx->launches += 1;
    CCHK(cudaGetLastError());
    return CS_OK;
}

cs_status cs_classifier_forward(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *xp,
                                float *logits_out) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_forward: unknown mesh id");
    if (n < 0 || (n > 0 && (!xp || !logits_out)))
        return fail(ctx, CS_EINVAL, "cs_classifier_forward: bad arguments");
    Classifier *C = get_cls(ctx, m->d.dim);
    if (!C) return fail(ctx, CS_ENOPRED, "cs_classifier_forward: no classifier loaded");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    cs_status rc = forward_chunks(ctx, *C, m->d, n, xp, logits_out, nullptr,
                                  [](int64_t, int64_t, const float *) { return CS_OK; });
    if (rc) return rc;
    CCHK(cudaGetLastError());
    return cs_device_status(ctx);     // synchronises
}

cs_status cs_classifier_labels(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *xp,
                               const int32_t *host, int32_t *label_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_labels: unknown mesh id");
    if (n < 0 || (n > 0 && (!xp || !host || !label_out)))
        return fail(ctx, CS_EINVAL, "cs_classifier_labels: bad arguments");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    launch_cls_labels(m->d, n, xp, host, label_out, ctx->sm_count,
                      static_cast<cudaStream_t>(stream));
    ctx->launches += 1;
    CCHK(cudaGetLastError());
    return CS_OK;
}

cs_status cs_classifier_pairs(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *x,
                              const double *u, double dt, const int32_t *start, double *xp_out,
                              int32_t *label_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_pairs: unknown mesh id");
    if (n < 0 || n >= (int64_t(1) << 31) - 1 || (n > 0 && (!x || !u || !xp_out || !label_out)))
        return fail(ctx, CS_EINVAL, "cs_classifier_pairs: bad arguments");
    if (!start && n != m->d.n_v)
        return fail(ctx, CS_EINVAL, "cs_classifier_pairs: start == NULL needs n == n_vertices");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the walk's outputs: host into label_out (overwritten by the labels),
    // path lengths and status into a scratch block
    void *scratch = nullptr;
    cs_status rc = dmalloc(ctx, &scratch, size_t(n) * 5);
    if (rc) return rc;
    int32_t *path = static_cast<int32_t *>(scratch);
    uint8_t *status = reinterpret_cast<uint8_t *>(path + n);
    rc = cs_track_impl(ctx, m, n, x, u, dt, start, CS_SNS, nullptr, label_out, path, status,
                       nullptr, st);
    if (rc == CS_OK) {
        launch_departure(n, m->d.dim, x, u, dt, xp_out, ctx->sm_count, st);
        launch_cls_labels(m->d, n, xp_out, label_out, label_out, ctx->sm_count, st);
        ctx->launches += 2;
        if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
            rc = fail(ctx, CS_ECUDA, "cs_classifier_pairs: kernel failed");
    }
    dfree(ctx, scratch);
    return rc;
}

cs_status cs_classifier_grad(cs_ctx *ctx, int32_t mesh_id, int64_t B, const double *xp,
                             const int32_t *labels, float *grad_out, float *loss_out) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_grad: unknown mesh id");
    if (B < 1 || !xp || !labels || !grad_out)
        return fail(ctx, CS_EINVAL, "cs_classifier_grad: bad arguments");
    Classifier *C = get_cls(ctx, m->d.dim);
    if (!C) return fail(ctx, CS_ENOPRED, "cs_classifier_grad: no classifier loaded");
    CCHK(cudaSetDevice(ctx->device));
    const bool tiled = tiled_batch(B);
    WorkspaceScope use;
    cs_status rc = with_room(ctx, *C, [&] {
        return tiled ? ensure_train(ctx, *C, B) : ensure_ws(ctx, *C, B, kWsAll);
    });
    if (rc) return rc;
    if (tiled) {
        ctx->launches += train_tiled(ctx, *C, m->d, B, xp, labels, nullptr, C->loss, nullptr);
    } else {
        CCHK(cudaMemset(C->loss, 0, sizeof(float)));
        ctx->launches += forward(ctx, *C, m->d, B, xp, nullptr, nullptr);
        ctx->launches += backward(ctx, *C, B, labels, nullptr, C->loss, nullptr);
    }
    CCHK(cudaGetLastError());
    if ((rc = cs_device_status(ctx))) return rc;     // synchronises
    CCHK(cudaMemcpyAsync(grad_out, C->g, size_t(C->n) * sizeof(float), cudaMemcpyDeviceToDevice,
                         nullptr));
    if (loss_out)
        CCHK(cudaMemcpy(loss_out, C->loss, sizeof(float), cudaMemcpyDeviceToHost));
    else
        CCHK(cudaDeviceSynchronize());
    return CS_OK;
}

cs_status cs_classifier_train(cs_ctx *ctx, int32_t mesh_id, const double *xp,
                              const int32_t *labels, int64_t N, int64_t batch, int64_t steps,
                              float lr, uint64_t seed, float *loss_out) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_train: unknown mesh id");
    if (!xp || !labels || N < 1 || batch < 1 || steps < 0 || !(lr > 0.f))
        return fail(ctx, CS_EINVAL, "cs_classifier_train: bad arguments");
    Classifier *C = get_cls(ctx, m->d.dim);
    if (!C) return fail(ctx, CS_ENOPRED, "cs_classifier_train: no classifier loaded");
    CCHK(cudaSetDevice(ctx->device));
    const int64_t B = std::min(batch, N);
    const bool tiled = tiled_batch(B);
    WorkspaceScope use;
    cs_status rc = with_room(ctx, *C, [&] {
        return tiled ? ensure_train(ctx, *C, B) : ensure_ws(ctx, *C, B, kWsAll);
    });
    if (rc) return rc;
    float *losses = nullptr;
    if ((rc = dmalloc_n(ctx, &losses, size_t(std::max<int64_t>(steps, 1))))) return rc;
    cs_status out = CS_OK;
    if (cudaMemset(losses, 0, size_t(std::max<int64_t>(steps, 1)) * sizeof(float)) != cudaSuccess)
        out = fail(ctx, CS_ECUDA, "cs_classifier_train: memset");
    std::vector<int64_t> perm(static_cast<size_t>(N));
    for (int64_t i = 0; i < N; ++i) perm[i] = i;
    uint64_t rs = seed;
    int64_t pos = N;   // shuffle at the first step
    std::vector<int64_t> idx(static_cast<size_t>(B));
    for (int64_t s = 0; s < steps && out == CS_OK; ++s) {
        for (int64_t b = 0; b < B; ++b) {
            if (pos >= N) {   // new epoch: Fisher-Yates shuffle
                for (int64_t i = N - 1; i > 0; --i) std::swap(perm[i], perm[splitmix(rs) % (i + 1)]);
                pos = 0;
            }
            idx[b] = perm[pos++];
        }
        int64_t *didx = tiled ? C->tidx : C->idx;
        if (cudaMemcpy(didx, idx.data(), size_t(B) * sizeof(int64_t), cudaMemcpyHostToDevice) !=
            cudaSuccess) {
            out = fail(ctx, CS_ECUDA, "cs_classifier_train: index copy");
            break;
        }
        if (tiled) {
            ctx->launches += train_tiled(ctx, *C, m->d, B, xp, labels, didx, losses + s, nullptr);
        } else {
            ctx->launches += forward(ctx, *C, m->d, B, xp, didx, nullptr);
            ctx->launches += backward(ctx, *C, B, labels, didx, losses + s, nullptr);
        }
        C->t += 1;
        ctx->launches += launch_adam(C->w, C->g, C->m, C->v, C->n, lr, C->t, ctx->dev_err,
                                     ctx->sm_count, nullptr);
        C->packed_dirty = true;
    }
    if (out == CS_OK) {
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (e == cudaSuccess && loss_out && steps > 0)
            e = cudaMemcpy(loss_out, losses, size_t(steps) * sizeof(float), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess)
            out = fail(ctx, CS_ECUDA, std::string("cs_classifier_train: ") + cudaGetErrorString(e));
        else
            out = cs_device_status(ctx);
    }
    dfree(ctx, losses);
    return out;
}

cs_status cs_classifier_start(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *xp,
                              const float *logits, const int32_t *fallback, int32_t *start_out,
                              int32_t *class_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_classifier_start: unknown mesh id");
    if (n < 0 || (n > 0 && (!xp || !logits || !start_out)))
        return fail(ctx, CS_EINVAL, "cs_classifier_start: bad arguments");
    if (!fallback && n != m->d.n_v)
        return fail(ctx, CS_EINVAL, "cs_classifier_start: fallback == NULL needs n == n_vertices");
    if (n == 0) return CS_OK;
    CCHK(cudaSetDevice(ctx->device));
    launch_cls_start(m->d, n, xp, logits, fallback, 0, start_out, class_out, ctx->sm_count,
                     static_cast<cudaStream_t>(stream));
    ctx->launches += 1;
    CCHK(cudaGetLastError());
    return CS_OK;
}

cs_status cs_track_classifier(cs_ctx *ctx, int32_t mesh_id, int64_t n, const double *x,
                              const double *u, double dt, const int32_t *start,
                              int32_t *host_out, int32_t *path_len_out, uint8_t *status_out,
                              int32_t *start_out, void *stream) {
    if (!ctx) return CS_EINVAL;
    cs::Mesh *m = find_mesh(ctx, mesh_id);
    if (!m) return fail(ctx, CS_ENOMESH, "cs_track_classifier: unknown mesh id");
    if (n < 0 || n >= (int64_t(1) << 31) - 1)
        return fail(ctx, CS_EINVAL, "cs_track_classifier: n is outside [0, 2^31 - 2]");
    Classifier *C = get_cls(ctx, m->d.dim);
    if (!C) return fail(ctx, CS_ENOPRED, "cs_track_classifier: no classifier loaded");
    if (n == 0) return CS_OK;
    if (!x || !u || !host_out || !path_len_out || !status_out)
        return fail(ctx, CS_EINVAL, "cs_track_classifier: null pointer");
    if (!start && n != m->d.n_v)
        return fail(ctx, CS_EINVAL, "cs_track_classifier: start == NULL needs n == n_vertices");
    CCHK(cudaSetDevice(ctx->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cs_status rc = ensure_xp(ctx, *C, n);
    if (rc) return rc;
    launch_departure(n, C->dim, x, u, dt, C->xp, ctx->sm_count, st);
    ctx->launches += 1;
    const DevMesh &d = m->d;
    rc = forward_chunks(ctx, *C, d, n, C->xp, nullptr, st, [&](int64_t r0, int64_t B, const float *H) {
        launch_cls_start(d, B, C->xp + r0 * C->dim, H, start ? start + r0 : nullptr, r0,
                         C->starts + r0, nullptr, ctx->sm_count, st);
        ctx->launches += 1;
        return CS_OK;
    });
    if (rc) return rc;
    rc = cs_track_impl(ctx, m, n, x, u, dt, C->starts, CS_SNS, nullptr, host_out, path_len_out,
                       status_out, nullptr, st);
    if (rc) return rc;
    if (start_out &&
        cudaMemcpyAsync(start_out, C->starts, size_t(n) * sizeof(int32_t), cudaMemcpyDeviceToDevice,
                        st) != cudaSuccess)
        return fail(ctx, CS_ECUDA, "cs_track_classifier: copy of the starts failed");
    CCHK(cudaStreamSynchronize(st));
    return cs_device_status(ctx);
}

}  // extern "C"
