// farm_mlp_api.cu -- the learned descriptor prefilter: weights, training on
// the GPU, loss/gradient evaluation, and tensor-core inference.
//
// f(x) = normalize(W2 gelu(W1 x + b1) + b2) maps a unit descriptor or query
// row (length D) to a unit vector of length P (128 by default).  Trained on
// (query row, object descriptor, oracle cosine y) pairs with the weighted
// squared error of f(q).f(d) against y, it replaces the full-length similarity
// stage by a P-length one whose best candidates are then re-scored exactly in
// FP32 (the plain full-descriptor path stays the fallback and the judge of
// its recall).  Training runs every contraction of the forward and backward
// passes as BF16 tensor-core products with FP32 accumulation (FP32 master
// weights, Adam); inference runs both layers the same way.  The FP32
// CUDA-core forward and backward are the reference arithmetic of
// farm_mlp_loss_grad and farm_mlp_embed.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "farm_internal.h"

using farm::Ctx;
using farm::Mlp;

namespace {

farm_status fail(Ctx &c, farm_status st, const std::string &msg)
{
    c.err = msg;
    return st;
}

#define MCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return fail(c, e_ == cudaErrorMemoryAllocation ? FARM_ENOMEM : FARM_ECUDA,             \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                       \
    } while (0)

#define MLAUNCH(call)     \
    do {                  \
        c.launches += 1;  \
        MCK(call);        \
    } while (0)

constexpr int64_t kEmbedChunk = 16384;   // rows per inference chunk

// SplitMix64 (Steele, Lea, Flood 2014) for the per-epoch shuffle.
uint64_t splitmix64(uint64_t &x)
{
    uint64_t z = (x += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Device scratch for training and loss/gradient evaluation (one allocation).
struct TrainBufs {
    float *base = nullptr;
    float *xq, *xd, *hq, *hd, *aq, *ad, *zq, *zd, *eq, *ed, *nq, *nd, *da, *grad, *m, *v, *loss, *y, *w;
};

cudaError_t train_alloc(farm_ctx *ctx, TrainBufs &t, const Mlp &M, int64_t B, int64_t loss_slots)
{
    const int64_t D = M.D, H = M.H, P = M.P, cnt = M.count();
    const int64_t sizes[] = {B * D, B * D, B * H, B * H, B * H, B * H, B * P, B * P, B * P, B * P,
                             B,     B,     B * H, cnt,   cnt,   cnt,   loss_slots, B, B};
    float **dst[] = {&t.xq, &t.xd, &t.hq, &t.hd, &t.aq, &t.ad, &t.zq, &t.zd, &t.eq, &t.ed,
                     &t.nq, &t.nd, &t.da, &t.grad, &t.m, &t.v, &t.loss, &t.y, &t.w};
    auto rounded = [](int64_t n) { return (n + 63) / 64 * 64; };   // 256-byte aligned sub-arrays
    int64_t total = 0;
    for (int64_t n : sizes) total += rounded(n);
    cudaError_t e = farm::dev_alloc(ctx, &t.base, (size_t)total * sizeof(float));
    if (e != cudaSuccess) return e;
    float *p = t.base;
    for (size_t i = 0; i < sizeof(sizes) / sizeof(sizes[0]); ++i) {
        *dst[i] = p;
        p += rounded(sizes[i]);
    }
    return cudaSuccess;
}

// Forward of b rows X [b, D] (lda D): h, a, z kept, e = f(X), norm.
cudaError_t forward(const Mlp &M, const float *X, int64_t b, float *h, float *a, float *z, float *e, float *nrm,
                    cudaStream_t s, int64_t &launches)
{
    cudaError_t r;
    launches += 4;
    if ((r = farm::mlp_gemm(false, false, (int)b, M.H, M.D, 1.f, X, M.D, M.W1(), M.D, 0.f, h, M.H, s))) return r;
    if ((r = farm::mlp_bias_gelu(h, M.b1(), a, b, M.H, s))) return r;
    if ((r = farm::mlp_gemm(false, false, (int)b, M.P, M.H, 1.f, a, M.H, M.W2(), M.H, 0.f, z, M.P, s))) return r;
    return farm::mlp_bias_normalize(z, M.b2(), e, nrm, b, M.P, s);
}

// Backward of one tower given de (overwritten) into grad (beta 0: set, 1: add).
cudaError_t backward(const Mlp &M, const float *X, int64_t b, float *h, const float *a, const float *e,
                     const float *nrm, float *de, float *da, float *grad, float beta, cudaStream_t s,
                     int64_t &launches)
{
    const int64_t D = M.D, H = M.H, P = M.P;
    float *gW1 = grad, *gb1 = grad + H * D, *gW2 = gb1 + H, *gb2 = gW2 + P * H;
    cudaError_t r;
    launches += 8;
    if ((r = farm::mlp_normalize_backward(e, nrm, de, b, (int)P, s))) return r;
    if ((r = farm::mlp_gemm(true, true, (int)P, (int)H, (int)b, 1.f, de, (int)P, a, (int)H, beta, gW2, (int)H, s)))
        return r;
    if ((r = farm::mlp_colsum(de, b, (int)P, gb2, beta != 0.f, s))) return r;
    if ((r = farm::mlp_gemm(false, true, (int)b, (int)H, (int)P, 1.f, de, (int)P, M.W2(), (int)H, 0.f, da, (int)H, s)))
        return r;
    if ((r = farm::mlp_gelu_backward(h, da, b * H, s))) return r;
    if ((r = farm::mlp_gemm(true, true, (int)H, (int)D, (int)b, 1.f, da, (int)H, X, (int)D, beta, gW1, (int)D, s)))
        return r;
    return farm::mlp_colsum(da, b, (int)H, gb1, beta != 0.f, s);
}

farm::MlpShape shape_of(const Mlp &M) { return {M.D, M.H, M.P, M.D_pad, M.w1b, M.w2b, M.w2t}; }

// BF16 copies of the weights for the tensor-core products: W1 padded to D_pad
// columns, W2, and W2 transposed ([H, P], the operand of the backward pass).
cudaError_t refresh_bf16_weights(Ctx &c)
{
    Mlp &M = c.mlp;
    c.launches += 1;
    M.version += 1;
    return farm::mlp_weights_bf16(M.params, M.count(), shape_of(M), c.stream);
}

// Device buffers of one tensor-core training step over up to B pairs: the
// two towers' rows are stacked (query rows 0..b-1, descriptor rows b..2b-1),
// so each contraction is one launch over them; the weight gradients contract
// over those rows (K), padded with zero columns to a multiple of 64.  dT
// holds dz^T (P rows), then dh^T (H rows): the operand rows of both weight
// gradients, computed by one launch.
struct TcBufs {
    void *base = nullptr;
    int64_t B = 0, K_pad = 0;
    uint16_t *x, *ab, *dzb, *xT, *aT, *dT;
    float *h, *z, *dz, *da, *grad, *m, *v, *loss, *y, *w, *bpart, *bdone;    // (bdone: counts, as int32)
    uint8_t *blob;               // the contractions' pieces, then their B tensor maps
};

int64_t round64(int64_t x) { return (x + 63) / 64 * 64; }

// The step's contractions: H = x W1^T, Z = a W2^T, dA = dz W2, and the two
// weight gradients.
enum { G_H = 0, G_Z, G_DA, G_DW, G_COUNT };
constexpr int kGemmPieces = 5;   // the weight gradients are two pieces
constexpr size_t kBlobMaps = 512;
static_assert(kGemmPieces * sizeof(farm::GemmPiece) <= kBlobMaps && kBlobMaps % 128 == 0, "piece table");
constexpr size_t kBlobBytes = kBlobMaps + kGemmPieces * 2 * farm::kTensorMapBytes;

// CTA pairs where their tiles occupy most of the chip, else 128 x 64 tiles: at
// 8,192 rows, D = 1152 the weight gradients (128 x 512 and 512 x 1152,
// contracting over the 8,192 rows) are 12 pair tiles and 80 narrow ones, and a
// step's contractions took 143 us with the pairs alone, 82 us with this rule.
// Every variant sums each output's products in the same order.
int gemm_variant(int64_t rows, int64_t n, int num_sms)
{
    return farm::sim_cluster_tiles(rows, n, farm::kSimPairVariant) * 8 >= (int64_t)num_sms * 3 ? farm::kSimPairVariant
                                                                                               : farm::kSimNarrowVariant;
}

struct GemmShape { int64_t rows, n; const uint16_t *b; int32_t k; float *out; int piece0, pieces; };

void gemm_shapes(const TcBufs &t, const Mlp &M, GemmShape (&g)[kGemmPieces])
{
    const int64_t R = 2 * t.B;
    float *gW1 = t.grad, *gW2 = t.grad + (int64_t)M.H * M.D + M.H;
    g[0] = {R, M.H, M.w1b, M.D_pad, t.h, 0, 1};
    g[1] = {R, M.P, M.w2b, M.H, t.z, 1, 1};
    g[2] = {R, M.H, M.w2t, M.P, t.da, 2, 1};
    g[3] = {M.P, M.H, t.aT, (int32_t)t.K_pad, gW2, 3, 2};
    g[4] = {M.H, M.D, t.xT, (int32_t)t.K_pad, gW1, 3, 2};
}

// Buffers of a training call up to this size stay with the context for its next
// one (allocating and freeing them takes longer than a few steps); they are
// given back by farm_memory_release, by farm_destroy, and to any allocation of
// the context that would fail otherwise.
constexpr int64_t kTrainKept = int64_t(512) << 20;

// keep: the buffers may be the context's kept ones (t.base then stays null).
cudaError_t tc_alloc(farm_ctx *ctx, TcBufs &t, int64_t B, int64_t loss_slots, bool keep)
{
    Ctx &c = *farm::ctx_of(ctx);
    const Mlp &M = c.mlp;
    const int64_t R = 2 * B, K = round64(2 * B), Dp = M.D_pad, H = M.H, P = M.P, cnt = M.count();
    t.B = B;
    t.K_pad = K;
    // (element count, element bytes) of each array, 256-byte aligned in one allocation
    const int64_t n16[] = {R * Dp, R * H, R * P, Dp * K, H * K, (P + H) * K};
    uint16_t **d16[] = {&t.x, &t.ab, &t.dzb, &t.xT, &t.aT, &t.dT};
    const int64_t n32[] = {R * H, R * P, R * P, R * H, cnt, cnt, cnt, loss_slots, B, B,
                           farm::bias_part_floats(K, H, P), farm::bias_blocks(H, P)};
    float **d32[] = {&t.h, &t.z, &t.dz, &t.da, &t.grad, &t.m, &t.v, &t.loss, &t.y, &t.w, &t.bpart, &t.bdone};
    auto al = [](int64_t bytes) { return (bytes + 255) / 256 * 256; };
    int64_t total = 0;
    for (int64_t n : n16) total += al(n * 2);
    for (int64_t n : n32) total += al(n * 4);
    total += (int64_t)kBlobBytes;
    void *at = nullptr;
    cudaError_t e;
    if (keep && total <= kTrainKept) {
        if ((e = farm::ws_alloc(ctx, farm::B_TRAIN, (size_t)total, &at)) != cudaSuccess) return e;
    } else {
        if ((e = farm::dev_alloc(ctx, &t.base, (size_t)total)) != cudaSuccess) return e;
        at = t.base;
    }
    char *p = static_cast<char *>(at);
    for (size_t i = 0; i < sizeof(n16) / sizeof(n16[0]); ++i) { *d16[i] = reinterpret_cast<uint16_t *>(p); p += al(n16[i] * 2); }
    for (size_t i = 0; i < sizeof(n32) / sizeof(n32[0]); ++i) { *d32[i] = reinterpret_cast<float *>(p); p += al(n32[i] * 4); }
    t.blob = reinterpret_cast<uint8_t *>(p);
    // (rows past a partial batch hold the last batch's, or zeros: every
    // contraction over them is finite and read by nothing)
    if ((e = cudaMemsetAsync(at, 0, (size_t)total, c.stream))) return e;
    GemmShape g[kGemmPieces];
    gemm_shapes(t, M, g);
    alignas(128) uint8_t host[kBlobBytes] = {};
    for (int k = 0; k < kGemmPieces; ++k) {
        const GemmShape &s = g[k];
        const int v = k >= G_DW ? farm::kSimNarrowVariant : gemm_variant(s.rows, s.n, c.num_sms);
        farm::GemmPiece gp{};
        gp.q_row0 = k == 4 ? P : 0;
        gp.s_off = k >= G_DW ? s.out - t.grad : 0;
        gp.tops_off = -1;
        gp.bmap = t.blob + kBlobMaps + (size_t)k * 2 * farm::kTensorMapBytes;
        gp.rows = (int32_t)s.rows;
        gp.n = gp.n_store = (int32_t)s.n;
        gp.ld = (int32_t)s.n;
        gp.tile_begin = k == 4 ? (int32_t)farm::sim_cluster_tiles(g[3].rows, g[3].n, farm::kSimNarrowVariant) : 0;
        gp.gshift = farm::kGroupShift;
        gp.col_mode = farm::kColAll;
        std::memcpy(host + k * sizeof(gp), &gp, sizeof(gp));
        if (!farm::sim_tc_encode_b(farm::kSimBf16, v,
                                   host + kBlobMaps + (size_t)k * 2 * farm::kTensorMapBytes, s.b, nullptr, s.n, s.k))
            return cudaErrorInvalidValue;
    }
    // (pageable source: staged when the call returns)
    return cudaMemcpyAsync(t.blob, host, kBlobBytes, cudaMemcpyHostToDevice, c.stream);
}

cudaError_t tc_gemm(Ctx &c, const TcBufs &t, int which)
{
    GemmShape g[kGemmPieces];
    gemm_shapes(t, c.mlp, g);
    const GemmShape &s = g[which];
    const bool dw = which == G_DW;
    const int v = dw ? farm::kSimNarrowVariant : gemm_variant(s.rows, s.n, c.num_sms);
    const uint16_t *a[] = {t.x, t.ab, t.dzb, t.dT};
    const int64_t rows = dw ? (int64_t)c.mlp.P + c.mlp.H : s.rows;
    int64_t tiles = 0;
    for (int k = s.piece0; k < s.piece0 + s.pieces; ++k) tiles += farm::sim_cluster_tiles(g[k].rows, g[k].n, v);
    return farm::launch_sim_tc_grouped(farm::kSimBf16, v, a[which], nullptr, rows, s.k,
                                       reinterpret_cast<const farm::GemmPiece *>(t.blob) + s.piece0, s.pieces, tiles,
                                       dw ? t.grad : s.out, nullptr, nullptr, c.num_sms, c.d_err, c.stream);
}

// Loss and gradient of b pairs, those at places off .. of the epoch's order
// (pairs.perm; null: pairs off .. themselves): their stacked BF16 input rows
// gathered, or already in t.x (pairs.row null); wsum the sum of their weights.
// The loss is added to *lslot, the gradient [W1 | b1 | W2 | b2] written to
// t.grad.
cudaError_t tc_loss_grad(Ctx &c, TcBufs &t, int64_t b, const farm::TrainPairs &pairs, int64_t off, float wsum,
                         float *lslot, int64_t &launches)
{
    const Mlp &M = c.mlp;
    const int64_t R = 2 * b, K = t.K_pad, H = M.H, P = M.P, D = M.D;
    float *gb1 = t.grad + H * D, *gb2 = gb1 + H + P * H;
    cudaStream_t st = c.stream;
    cudaError_t r;
    launches += 8;
    if ((r = farm::mlp_train_rows(pairs, off, b, (int)D, M.D_pad, t.x, t.xT, K, st))) return r;
    // forward: h = x W1^T, a = gelu(h + b1), z = a W2^T
    if ((r = tc_gemm(c, t, G_H))) return r;
    if ((r = farm::mlp_gelu_bf16(t.h, M.b1(), R, (int)H, t.ab, t.aT, K, st))) return r;
    if ((r = tc_gemm(c, t, G_Z))) return r;
    // e = (z + b2) / |z + b2|, the loss and dz
    if ((r = farm::mlp_pair_step(t.z, M.b2(), pairs, off, wsum, b, (int)P, t.dz, t.dzb, t.dT, K, lslot, st))) return r;
    // backward: da = dz W2, dh = gelu'(h + b1) da and the bias sums, then dW2 = dz^T a and dW1 = dh^T x together
    if ((r = tc_gemm(c, t, G_DA))) return r;
    if ((r = farm::mlp_gelu_backward_t(t.h, M.b1(), t.da, R, (int)H, t.dT + P * K, K, gb1, t.dz, (int)P, gb2,
                                       t.bpart, reinterpret_cast<int32_t *>(t.bdone), st))) return r;
    return tc_gemm(c, t, G_DW);
}

}  // namespace

namespace {

cudaError_t embed_buffers(farm_ctx *ctx, int64_t rows, void **h, void **ab, void **z)
{
    const Mlp &M = farm::ctx_of(ctx)->mlp;
    const int64_t chunk = std::max<int64_t>(1, std::min<int64_t>(rows, kEmbedChunk));
    cudaError_t r;
    if ((r = farm::ws_alloc(ctx, farm::B_MLP_H, (size_t)chunk * M.H * 4, h))) return r;
    if ((r = farm::ws_alloc(ctx, farm::B_MLP_AB, (size_t)chunk * M.H * 2, ab))) return r;
    return farm::ws_alloc(ctx, farm::B_MLP_Z, (size_t)chunk * M.P * 4, z);
}

}  // namespace

cudaError_t farm::learned_reserve(farm_ctx *ctx, int64_t rows)
{
    void *h, *ab, *z;
    return embed_buffers(ctx, rows, &h, &ab, &z);
}

cudaError_t farm::learned_embed_rows(farm_ctx *ctx, const uint16_t *xb, int64_t rows, uint16_t *out)
{
    Ctx &c = *ctx_of(ctx);
    const Mlp &M = c.mlp;
    const int64_t chunk = std::min<int64_t>(rows, kEmbedChunk);
    void *h, *ab, *z;
    cudaError_t r;
    if ((r = embed_buffers(ctx, rows, &h, &ab, &z))) return r;
    for (int64_t r0 = 0; r0 < rows; r0 += chunk) {
        const int64_t b = std::min(chunk, rows - r0);
        c.launches += 4;
        if ((r = launch_sim_tc_bf16(xb + r0 * M.D_pad, M.w1b, (float *)h, b, M.H, M.D_pad, M.H, nullptr, c.num_sms, c.d_err,
                                    c.stream)))
            return r;
        if ((r = mlp_gelu_bf16((float *)h, M.b1(), b, M.H, (uint16_t *)ab, nullptr, 0, c.stream))) return r;
        if ((r = launch_sim_tc_bf16((uint16_t *)ab, M.w2b, (float *)z, b, M.P, M.H, M.P, nullptr, c.num_sms, c.d_err,
                                    c.stream)))
            return r;
        if ((r = mlp_normalize_bf16((float *)z, M.b2(), b, M.P, out + r0 * M.P, c.stream))) return r;
    }
    return cudaSuccess;
}

cudaError_t farm::learned_refresh_scene(farm_ctx *ctx, int32_t scene_id)
{
    Ctx &c = *ctx_of(ctx);
    Scene &s = c.scenes[scene_id];
    if (s.comp && s.comp_version == c.mlp.version) return cudaSuccess;
    cudaError_t r;
    if (!s.comp) {
        if ((r = cudaStreamSynchronize(c.stream))) return r;
        if ((r = farm::dev_alloc(ctx, &s.comp, (size_t)s.n * c.mlp.P * 2))) return r;
    }
    if ((r = learned_embed_rows(ctx, s.desc_bf16, s.n, s.comp))) return r;
    s.comp_version = c.mlp.version;
    return cudaSuccess;
}

extern "C" {

farm_status farm_mlp_set(farm_ctx *ctx, int32_t dim, int32_t hidden, int32_t out_dim, const float *W1,
                         const float *b1, const float *W2, const float *b2)
{
    if (!ctx) return FARM_EINVAL;
    Ctx &c = *farm::ctx_of(ctx);
    if (dim < 1 || dim > 8192 || hidden < 64 || hidden > 4096 || hidden % 64 || out_dim < 64 || out_dim > 1024 ||
        out_dim % 64)
        return fail(c, FARM_EINVAL, "farm_mlp_set: need 1 <= dim <= 8192, hidden in [64, 4096] and out_dim in "
                                    "[64, 1024], both multiples of 64");
    if (!W1 || !b1 || !W2 || !b2) return fail(c, FARM_EINVAL, "farm_mlp_set: weights must be non-null");
    MCK(cudaSetDevice(c.device));
    Mlp &M = c.mlp;
    Mlp nm;
    nm.D = dim; nm.H = hidden; nm.P = out_dim;
    nm.D_pad = (dim + farm::kDimAlign - 1) / farm::kDimAlign * farm::kDimAlign;
    const int64_t cnt = nm.count();
    const float *part[4] = {W1, b1, W2, b2};
    const size_t len[4] = {(size_t)nm.H * nm.D, (size_t)nm.H, (size_t)nm.P * nm.H, (size_t)nm.P};
    for (int k = 0; k < 4; ++k) {
        uint32_t bad = 0;                 // (branch-free: the loop vectorises)
        for (size_t i = 0; i < len[k]; ++i) {
            uint32_t u;
            std::memcpy(&u, part[k] + i, 4);
            bad |= (u & 0x7f800000u) == 0x7f800000u ? 1u : 0u;
        }
        if (bad) return fail(c, FARM_EINVAL, "farm_mlp_set: non-finite weight");
    }
    MCK(cudaStreamSynchronize(c.stream));
    if (M.set && (M.D != nm.D || M.H != nm.H || M.P != nm.P)) {
        cudaFree(M.params); cudaFree(M.w1b); cudaFree(M.w2b); cudaFree(M.w2t);
        M.params = nullptr; M.w1b = nullptr; M.w2b = nullptr; M.w2t = nullptr;
        M.set = false;
    }
    if (!M.set) {
        MCK(farm::dev_alloc(ctx, &M.params, (size_t)cnt * 4));
        MCK(farm::dev_alloc(ctx, &M.w1b, (size_t)nm.H * nm.D_pad * 2));
        MCK(farm::dev_alloc(ctx, &M.w2b, (size_t)nm.P * nm.H * 2));
        MCK(farm::dev_alloc(ctx, &M.w2t, (size_t)nm.H * nm.P * 2));
        M.D = nm.D; M.H = nm.H; M.P = nm.P; M.D_pad = nm.D_pad;
        // shape change: every scene cache is stale
        for (auto &s : c.scenes)
            if (s.comp) { cudaFree(s.comp); s.comp = nullptr; }
    }
    float *to = M.params;
    for (int k = 0; k < 4; ++k) {
        MCK(cudaMemcpyAsync(to, part[k], len[k] * 4, cudaMemcpyHostToDevice, c.stream));
        to += len[k];
    }
    M.set = true;
    MCK(refresh_bf16_weights(c));
    // the caller's arrays must have been read before the call returns
    MCK(cudaStreamSynchronize(c.stream));
    return FARM_OK;
}

farm_status farm_mlp_get(farm_ctx *ctx, float *W1, float *b1, float *W2, float *b2)
{
    if (!ctx) return FARM_EINVAL;
    Ctx &c = *farm::ctx_of(ctx);
    const Mlp &M = c.mlp;
    if (!M.set) return fail(c, FARM_ESTATE, "farm_mlp_get: no weights set");
    MCK(cudaSetDevice(c.device));
    if (W1) MCK(cudaMemcpyAsync(W1, M.W1(), (size_t)M.H * M.D * 4, cudaMemcpyDeviceToHost, c.stream));
    if (b1) MCK(cudaMemcpyAsync(b1, M.b1(), (size_t)M.H * 4, cudaMemcpyDeviceToHost, c.stream));
    if (W2) MCK(cudaMemcpyAsync(W2, M.W2(), (size_t)M.P * M.H * 4, cudaMemcpyDeviceToHost, c.stream));
    if (b2) MCK(cudaMemcpyAsync(b2, M.b2(), (size_t)M.P * 4, cudaMemcpyDeviceToHost, c.stream));
    MCK(cudaStreamSynchronize(c.stream));
    return FARM_OK;
}

farm_status farm_mlp_loss_grad(farm_ctx *ctx, int64_t n_pairs, const float *xq, const float *xd, const float *y,
                               const float *w, int32_t precision, float *loss, float *grad)
{
    if (!ctx) return FARM_EINVAL;
    Ctx &c = *farm::ctx_of(ctx);
    const Mlp &M = c.mlp;
    if (!M.set) return fail(c, FARM_ESTATE, "farm_mlp_loss_grad: no weights set");
    if (n_pairs < 1 || n_pairs > (1 << 20) || !xq || !xd || !y || !loss)
        return fail(c, FARM_EINVAL, "farm_mlp_loss_grad: bad arguments");
    if (precision != FARM_PREC_FP32_SIMT && precision != FARM_PREC_BF16)
        return fail(c, FARM_EINVAL, "farm_mlp_loss_grad: precision must be FARM_PREC_FP32_SIMT or FARM_PREC_BF16");
    MCK(cudaSetDevice(c.device));
    double wsum = 0.0;
    for (int64_t i = 0; i < n_pairs; ++i) wsum += w ? (double)w[i] : 1.0;
    if (!(wsum > 0.0)) return fail(c, FARM_EINVAL, "farm_mlp_loss_grad: weights sum to zero");
    const size_t xb = (size_t)n_pairs * M.D * 4;
    int64_t L = 0;
    cudaError_t e = cudaSuccess;
    if (precision == FARM_PREC_BF16) {
        // the training step's arithmetic: stacked rows in BF16, tensor-core contractions
        TcBufs t;
        float *raw = nullptr;
        auto done = [&](farm_status st) { cudaStreamSynchronize(c.stream); cudaFree(t.base); cudaFree(raw); return st; };
        e = tc_alloc(ctx, t, n_pairs, 1, false);
        if (e) return done(fail(c, e == cudaErrorMemoryAllocation ? FARM_ENOMEM : FARM_ECUDA,
                                std::string("farm_mlp_loss_grad: ") + cudaGetErrorString(e)));
        if (!e) e = farm::dev_alloc(ctx, &raw, 2 * xb);
        if (!e) e = cudaMemcpyAsync(raw, xq, xb, cudaMemcpyHostToDevice, c.stream);
        if (!e) e = cudaMemcpyAsync(raw + (size_t)n_pairs * M.D, xd, xb, cudaMemcpyHostToDevice, c.stream);
        if (!e) e = cudaMemcpyAsync(t.y, y, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, c.stream);
        if (!e && w) e = cudaMemcpyAsync(t.w, w, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, c.stream);
        if (!e) e = cudaMemsetAsync(t.loss, 0, 4, c.stream);
        if (!e) e = farm::mlp_to_bf16_padded(raw, 2 * n_pairs, M.D, t.x, M.D_pad, c.stream);
        if (!e) e = tc_loss_grad(c, t, n_pairs,
                                 farm::TrainPairs{nullptr, 0, nullptr, nullptr, nullptr, t.y, w ? t.w : nullptr, nullptr},
                                 0, (float)wsum, t.loss, L);
        if (!e) e = cudaMemcpyAsync(loss, t.loss, 4, cudaMemcpyDeviceToHost, c.stream);
        if (!e && grad) e = cudaMemcpyAsync(grad, t.grad, (size_t)M.count() * 4, cudaMemcpyDeviceToHost, c.stream);
        if (!e) e = cudaStreamSynchronize(c.stream);
        c.launches += L + 1;
        if (e) return done(fail(c, FARM_ECUDA, std::string("farm_mlp_loss_grad: ") + cudaGetErrorString(e)));
        return done(FARM_OK);
    }
    TrainBufs t;
    MCK(train_alloc(ctx, t, M, n_pairs, 1));
    auto done = [&](farm_status st) { cudaFree(t.base); return st; };
    if (!e) e = cudaMemcpyAsync(t.xq, xq, xb, cudaMemcpyHostToDevice, c.stream);
    if (!e) e = cudaMemcpyAsync(t.xd, xd, xb, cudaMemcpyHostToDevice, c.stream);
    if (!e) e = cudaMemcpyAsync(t.y, y, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, c.stream);
    if (!e && w) e = cudaMemcpyAsync(t.w, w, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, c.stream);
    if (!e) e = cudaMemsetAsync(t.loss, 0, 4, c.stream);
    if (!e) e = forward(M, t.xq, n_pairs, t.hq, t.aq, t.zq, t.eq, t.nq, c.stream, L);
    if (!e) e = forward(M, t.xd, n_pairs, t.hd, t.ad, t.zd, t.ed, t.nd, c.stream, L);
    // de of both towers into zq / zd (the pre-normalisation values are no longer needed)
    if (!e) e = farm::mlp_pair_loss(t.eq, t.ed, t.y, w ? t.w : nullptr, (float)wsum, n_pairs, M.P, t.zq, t.zd,
                                    t.loss, c.stream);
    if (!e) e = backward(M, t.xq, n_pairs, t.hq, t.aq, t.eq, t.nq, t.zq, t.da, t.grad, 0.f, c.stream, L);
    if (!e) e = backward(M, t.xd, n_pairs, t.hd, t.ad, t.ed, t.nd, t.zd, t.da, t.grad, 1.f, c.stream, L);
    if (!e) e = cudaMemcpyAsync(loss, t.loss, 4, cudaMemcpyDeviceToHost, c.stream);
    if (!e && grad) e = cudaMemcpyAsync(grad, t.grad, (size_t)M.count() * 4, cudaMemcpyDeviceToHost, c.stream);
    if (!e) e = cudaStreamSynchronize(c.stream);
    c.launches += L + 1;
    if (e) return done(fail(c, FARM_ECUDA, std::string("farm_mlp_loss_grad: ") + cudaGetErrorString(e)));
    return done(FARM_OK);
}

farm_status farm_mlp_train(farm_ctx *ctx, int32_t n_scenes, const int32_t *scene_ids, int64_t n_rows,
                           const float *rows, int64_t n_pairs, const int32_t *pair_row, const int32_t *pair_scene,
                           const int32_t *pair_obj, const float *y, const float *w, int32_t epochs, int32_t batch,
                           float lr, uint64_t seed, float *loss_out)
{
    if (!ctx) return FARM_EINVAL;
    Ctx &c = *farm::ctx_of(ctx);
    Mlp &M = c.mlp;
    if (!M.set) return fail(c, FARM_ESTATE, "farm_mlp_train: set initial weights with farm_mlp_set first");
    if (n_scenes < 1 || n_scenes > 64 || !scene_ids || (n_scenes > 1 && !pair_scene))
        return fail(c, FARM_EINVAL, "farm_mlp_train: need 1..64 scene ids (and pair_scene for more than one)");
    std::vector<const uint16_t *> bases((size_t)n_scenes + 1);   // the scenes' BF16 descriptors, then the rows
    std::vector<int64_t> scene_n((size_t)n_scenes);
    for (int32_t k = 0; k < n_scenes; ++k) {
        const int32_t sid = scene_ids[k];
        if (sid < 0 || sid >= (int32_t)c.scenes.size() || !c.scenes[sid].present)
            return fail(c, FARM_EINVAL, "farm_mlp_train: unknown scene");
        const farm::Scene &s = c.scenes[sid];
        if (s.dim != M.D) return fail(c, FARM_EINVAL, "farm_mlp_train: scene dim differs from the network's");
        bases[k] = s.desc_bf16;
        scene_n[k] = s.n;
    }
    if (n_rows < 1 || !rows || n_pairs < 1 || !pair_row || !pair_obj || !y || epochs < 1 || batch < 1 ||
        batch > (1 << 16) || !(lr > 0.f))
        return fail(c, FARM_EINVAL, "farm_mlp_train: bad arguments");
    for (int64_t i = 0; i < n_pairs; ++i) {
        const int32_t k = pair_scene ? pair_scene[i] : 0;
        if (pair_row[i] < 0 || pair_row[i] >= n_rows || k < 0 || k >= n_scenes || pair_obj[i] < 0 ||
            pair_obj[i] >= scene_n[k] || !std::isfinite(y[i]) || (w && !(w[i] >= 0.f)))
            return fail(c, FARM_EINVAL, "farm_mlp_train: pair " + std::to_string(i) + " out of range");
    }
    MCK(cudaSetDevice(c.device));
    const int64_t B = std::min<int64_t>(batch, n_pairs);
    const int64_t steps = (n_pairs + B - 1) / B;
    TcBufs t;
    struct Busy {
        bool &b;
        explicit Busy(bool &x) : b(x) { b = true; }
        ~Busy() { b = false; }
    } busy(c.training);
    // the call's inputs: normalised rows (BF16 [n_rows, D_pad]), the rows as
    // given, the pairs' arrays as given, an epoch's order, the row tables
    uint16_t *qnb = nullptr;
    float *raw = nullptr, *d_y = nullptr, *d_w = nullptr;
    int32_t *d_row = nullptr, *d_obj = nullptr, *d_scene = nullptr, *d_perm = nullptr;
    const uint16_t **d_bases = nullptr;
    void *in_base = nullptr;       // the inputs' memory when it is this call's own
    auto done = [&](farm_status st) {
        cudaStreamSynchronize(c.stream);
        cudaFree(t.base); cudaFree(in_base);
        return st;
    };
    cudaError_t e = tc_alloc(ctx, t, B, steps * (int64_t)epochs, true);
    if (e) return done(fail(c, e == cudaErrorMemoryAllocation ? FARM_ENOMEM : FARM_ECUDA,
                            std::string("farm_mlp_train: ") + cudaGetErrorString(e)));
    {
        const size_t sizes[] = {(size_t)n_rows * M.D_pad * 2, (size_t)n_rows * M.D * 4, (size_t)n_pairs * 4,
                                (size_t)n_pairs * 4, (size_t)n_pairs * 4, (size_t)n_pairs * 4, (size_t)n_pairs * 4,
                                (size_t)n_pairs * 4, bases.size() * sizeof(void *)};
        void **to[] = {(void **)&qnb, (void **)&raw, (void **)&d_y, (void **)&d_w, (void **)&d_row, (void **)&d_obj,
                       (void **)&d_scene, (void **)&d_perm, (void **)&d_bases};
        size_t total = 0;
        for (size_t b : sizes) total += (b + 255) & ~size_t(255);
        void *at = nullptr;
        if ((int64_t)total <= kTrainKept) e = farm::ws_alloc(ctx, farm::B_TRAIN_IN, total, &at);
        else if (!(e = farm::dev_alloc(ctx, &in_base, total))) at = in_base;
        if (e) return done(fail(c, e == cudaErrorMemoryAllocation ? FARM_ENOMEM : FARM_ECUDA,
                                std::string("farm_mlp_train: ") + cudaGetErrorString(e)));
        uint8_t *p = static_cast<uint8_t *>(at);
        for (size_t k = 0; k < sizeof(sizes) / sizeof(sizes[0]); ++k) {
            *to[k] = p;
            p += (sizes[k] + 255) & ~size_t(255);
        }
        const cudaMemcpyKind h2d = cudaMemcpyHostToDevice;
        if (!e) e = cudaMemcpyAsync(d_y, y, (size_t)n_pairs * 4, h2d, c.stream);
        if (!e && w) e = cudaMemcpyAsync(d_w, w, (size_t)n_pairs * 4, h2d, c.stream);
        if (!e) e = cudaMemcpyAsync(d_row, pair_row, (size_t)n_pairs * 4, h2d, c.stream);
        if (!e) e = cudaMemcpyAsync(d_obj, pair_obj, (size_t)n_pairs * 4, h2d, c.stream);
        if (!e && pair_scene) e = cudaMemcpyAsync(d_scene, pair_scene, (size_t)n_pairs * 4, h2d, c.stream);
    }
    bases[n_scenes] = qnb;
    if (!e) e = cudaMemcpyAsync(d_bases, bases.data(), bases.size() * sizeof(void *), cudaMemcpyHostToDevice,
                                c.stream);
    if (!e) e = cudaMemcpyAsync(raw, rows, (size_t)n_rows * M.D * 4, cudaMemcpyHostToDevice, c.stream);
    if (!e) e = farm::launch_normalize_rows(raw, nullptr, n_rows, M.D, M.D_pad, nullptr, nullptr, nullptr, qnb,
                                            c.d_err, farm::kErrBadRow, c.stream);
    // (the moments and the losses start at zero: tc_alloc clears them)
    if (e) return done(fail(c, FARM_ECUDA, std::string("farm_mlp_train: ") + cudaGetErrorString(e)));
    std::vector<int32_t> perm((size_t)n_pairs);
    for (int64_t i = 0; i < n_pairs; ++i) perm[i] = (int32_t)i;
    const farm::TrainPairs pairs{d_bases, n_scenes, d_row, d_obj, pair_scene ? d_scene : nullptr, d_y,
                                 w ? d_w : nullptr, d_perm};
    uint64_t st = seed;
    int64_t L = 2;
    int t_adam = 0;
    for (int32_t ep = 0; ep < epochs && !e; ++ep) {
        for (int64_t i = n_pairs - 1; i > 0; --i) {
            const int64_t j = (int64_t)(splitmix64(st) % (uint64_t)(i + 1));
            std::swap(perm[i], perm[j]);
        }
        // the previous epoch's kernels may still read the device copy
        e = cudaStreamSynchronize(c.stream);
        if (!e) e = cudaMemcpyAsync(d_perm, perm.data(), (size_t)n_pairs * 4, cudaMemcpyHostToDevice, c.stream);
        for (int64_t sidx = 0; sidx < steps && !e; ++sidx) {
            const int64_t off = sidx * B;
            const int64_t b = std::min(B, n_pairs - off);
            double wsum = 0.0;
            if (w) {
                for (int64_t i = 0; i < b; ++i) wsum += w[perm[off + i]];
            } else {
                wsum = (double)b;
            }
            if (!(wsum > 0.0)) continue;
            float *lslot = t.loss + (int64_t)ep * steps + sidx;
            e = tc_loss_grad(c, t, b, pairs, off, (float)wsum, lslot, L);
            if (!e) e = farm::mlp_adam(M.params, t.grad, t.m, t.v, M.count(), lr, ++t_adam, shape_of(M), c.stream);
            M.version += 1;
            L += 1;
        }
    }
    c.launches += L;
    if (!e && loss_out) {
        std::vector<float> ls((size_t)steps * epochs);
        e = cudaMemcpyAsync(ls.data(), t.loss, ls.size() * 4, cudaMemcpyDeviceToHost, c.stream);
        if (!e) e = cudaStreamSynchronize(c.stream);
        for (int32_t ep = 0; ep < epochs && !e; ++ep) {
            double acc = 0.0;
            for (int64_t i = 0; i < steps; ++i) acc += ls[(size_t)ep * steps + i];
            loss_out[ep] = (float)(acc / (double)steps);
        }
    }
    if (e) return done(fail(c, FARM_ECUDA, std::string("farm_mlp_train: ") + cudaGetErrorString(e)));
    return done(FARM_OK);
}

farm_status farm_mlp_embed(farm_ctx *ctx, int64_t n_rows, const float *x, int32_t precision, float *out)
{
    if (!ctx) return FARM_EINVAL;
    Ctx &c = *farm::ctx_of(ctx);
    const Mlp &M = c.mlp;
    if (!M.set) return fail(c, FARM_ESTATE, "farm_mlp_embed: no weights set");
    if (n_rows < 0 || (n_rows > 0 && (!x || !out))) return fail(c, FARM_EINVAL, "farm_mlp_embed: bad arguments");
    if (precision != FARM_PREC_FP32_SIMT && precision != FARM_PREC_BF16)
        return fail(c, FARM_EINVAL, "farm_mlp_embed: precision must be FARM_PREC_FP32_SIMT or FARM_PREC_BF16");
    if (n_rows == 0) return FARM_OK;
    MCK(cudaSetDevice(c.device));
    float *raw = nullptr, *xn = nullptr, *h = nullptr, *a = nullptr, *z = nullptr, *e32 = nullptr;
    uint16_t *xb = nullptr, *eb = nullptr;
    auto done = [&](farm_status st) {
        cudaStreamSynchronize(c.stream);
        cudaFree(raw); cudaFree(xn); cudaFree(h); cudaFree(a); cudaFree(z); cudaFree(e32); cudaFree(xb); cudaFree(eb);
        return st;
    };
    cudaError_t e = farm::dev_alloc(ctx, &raw, (size_t)n_rows * M.D * 4);
    if (!e) e = cudaMemcpyAsync(raw, x, (size_t)n_rows * M.D * 4, cudaMemcpyHostToDevice, c.stream);
    if (precision == FARM_PREC_FP32_SIMT) {
        if (!e) e = farm::dev_alloc(ctx, &xn, (size_t)n_rows * M.D * 4);
        if (!e) e = farm::dev_alloc(ctx, &h, (size_t)n_rows * M.H * 4);
        if (!e) e = farm::dev_alloc(ctx, &a, (size_t)n_rows * M.H * 4);
        if (!e) e = farm::dev_alloc(ctx, &z, (size_t)n_rows * M.P * 4);
        if (!e) e = farm::dev_alloc(ctx, &e32, (size_t)n_rows * M.P * 4);
        if (!e) e = farm::launch_normalize_rows(raw, nullptr, n_rows, M.D, M.D, xn, nullptr, nullptr, nullptr, c.d_err,
                                                farm::kErrBadRow, c.stream);
        int64_t L = 1;
        if (!e) e = forward(M, xn, n_rows, h, a, z, e32, nullptr, c.stream, L);
        c.launches += L;
        if (!e) e = cudaMemcpyAsync(out, e32, (size_t)n_rows * M.P * 4, cudaMemcpyDeviceToHost, c.stream);
    } else {
        if (!e) e = farm::dev_alloc(ctx, &xb, (size_t)n_rows * M.D_pad * 2);
        if (!e) e = farm::dev_alloc(ctx, &eb, (size_t)n_rows * M.P * 2);
        if (!e) e = farm::dev_alloc(ctx, &e32, (size_t)n_rows * M.P * 4);
        if (!e) e = farm::launch_normalize_rows(raw, nullptr, n_rows, M.D, M.D_pad, nullptr, nullptr, nullptr, xb,
                                                c.d_err, farm::kErrBadRow, c.stream);
        c.launches += 1;
        if (!e) e = farm::learned_embed_rows(ctx, xb, n_rows, eb);
        // widen the BF16 embeddings for the caller
        std::vector<uint16_t> hb;
        if (!e) {
            hb.resize((size_t)n_rows * M.P);
            e = cudaMemcpyAsync(hb.data(), eb, hb.size() * 2, cudaMemcpyDeviceToHost, c.stream);
        }
        if (!e) e = cudaStreamSynchronize(c.stream);
        if (!e)
            for (size_t i = 0; i < hb.size(); ++i) {
                const uint32_t u = (uint32_t)hb[i] << 16;
                std::memcpy(out + i, &u, 4);
            }
    }
    if (!e) e = cudaStreamSynchronize(c.stream);
    if (e) return done(fail(c, FARM_ECUDA, std::string("farm_mlp_embed: ") + cudaGetErrorString(e)));
    farm_status st = FARM_OK;
    if (c.h_err) {
        cudaMemcpy(c.h_err, c.d_err, 4, cudaMemcpyDeviceToHost);
        if (*c.h_err) {
            cudaMemset(c.d_err, 0, 4);
            st = fail(c, FARM_EINVAL, "farm_mlp_embed: a row has zero or non-finite norm");
        }
    }
    return done(st);
}

}  // extern "C"
