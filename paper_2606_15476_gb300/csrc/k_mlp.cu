// k_mlp.cu -- kernels of the learned descriptor prefilter: a two-layer MLP
//   f(x) = normalize(W2 gelu(W1 x + b1) + b2),   x in R^D, W1: H x D, W2: P x H,
// its forward and backward passes for training on (query row, descriptor,
// oracle cosine) pairs with the loss
//   L = sum_i w_i (f(q_i) . f(d_i) - y_i)^2 / sum_i w_i,
// and an Adam update.  The contractions of training and inference run on the
// tensor cores (BF16 operands, FP32 accumulation) through the similarity
// kernel of k_sim_tc.cu, fed by the gathers, transposes and BF16 conversions
// below; the tiled FP32 GEMM on the CUDA cores here is the FP32 reference
// arithmetic of farm_mlp_loss_grad and farm_mlp_embed.  Elementwise steps
// (bias, GELU in its exact erf form, normalisation, the loss and their
// gradients, Adam) are FP32 on the CUDA cores.
#include <cuda_bf16.h>

#include "farm_internal.h"

namespace farm {
namespace {

// C[M,N] (ldc) = alpha * op(A) op(B) + beta * C.
//   TA = false: A is [M, K] (lda), K contiguous;  TA = true: A is [K, M] (lda), M contiguous.
//   TB = false: B is [N, K] (ldb), K contiguous;  TB = true: B is [K, N] (ldb), N contiguous.
// 64 x 64 tiles, 16-wide K slices, 256 threads with 4 x 4 outputs each; all
// bounds checked (M, N, K arbitrary).
template <bool TA, bool TB>
__global__ void __launch_bounds__(256)
gemm_f32_kernel(int M, int N, int K, float alpha, const float *__restrict__ A, int lda,
                const float *__restrict__ B, int ldb, float beta, float *__restrict__ C, int ldc)
{
    __shared__ float As[16][64 + 1];
    __shared__ float Bs[16][64 + 1];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int tx = tid & 15, ty = tid >> 4;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += 16) {
        // 64 x 16 elements per operand, 4 per thread
        for (int e = tid; e < 64 * 16; e += 256) {
            int mm, kk;
            if (TA) { mm = e & 63; kk = e >> 6; } else { kk = e & 15; mm = e >> 4; }
            const int gm = m0 + mm, gk = k0 + kk;
            float v = 0.f;
            if (gm < M && gk < K) v = TA ? A[(int64_t)gk * lda + gm] : A[(int64_t)gm * lda + gk];
            As[kk][mm] = v;
        }
        for (int e = tid; e < 64 * 16; e += 256) {
            int nn, kk;
            if (TB) { nn = e & 63; kk = e >> 6; } else { kk = e & 15; nn = e >> 4; }
            const int gn = n0 + nn, gk = k0 + kk;
            float v = 0.f;
            if (gn < N && gk < K) v = TB ? B[(int64_t)gk * ldb + gn] : B[(int64_t)gn * ldb + gk];
            Bs[kk][nn] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + ty * 4 + i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tx * 4 + j;
            if (gn >= N) continue;
            float *c = C + (int64_t)gm * ldc + gn;
            *c = alpha * acc[i][j] + (beta != 0.f ? beta * *c : 0.f);
        }
    }
}

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad(float x)
{
    const float cdf = 0.5f * (1.f + erff(x * 0.70710678118654752f));
    const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
    return cdf + x * pdf;
}

__device__ __forceinline__ uint16_t bf16_bits(float x)
{
    __nv_bfloat16 b = __float2bfloat16_rn(x);
    return *reinterpret_cast<uint16_t *>(&b);
}

// h[r, j] += b[j] (pre-activation kept), a[r, j] = gelu(h[r, j]).
__global__ void bias_gelu_kernel(float *__restrict__ h, const float *__restrict__ b, float *__restrict__ a,
                                 int64_t rows, int cols)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * cols) return;
    const float v = h[i] + b[i % cols];
    h[i] = v;
    a[i] = gelu(v);
}

// z[r, :] += b, then e = z / |z| (norm kept); one warp per row.
__global__ void bias_normalize_kernel(float *__restrict__ z, const float *__restrict__ b, float *__restrict__ e,
                                      float *__restrict__ norm, int64_t rows, int cols)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    float *zr = z + r * cols;
    float ss = 0.f;
    for (int j = lane; j < cols; j += 32) {
        const float v = zr[j] + b[j];
        zr[j] = v;
        ss = fmaf(v, v, ss);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float nrm = fmaxf(sqrtf(ss), 1e-20f);
    if (lane == 0 && norm) norm[r] = nrm;
    for (int j = lane; j < cols; j += 32) e[r * cols + j] = zr[j] / nrm;
}

// Per pair: s = eq . ed, loss += w (s - y)^2 / wsum, deq = g ed, ded = g eq
// with g = 2 w (s - y) / wsum.  One warp per pair.
__global__ void pair_loss_kernel(const float *__restrict__ eq, const float *__restrict__ ed,
                                 const float *__restrict__ y, const float *__restrict__ w, float wsum, int64_t pairs,
                                 int cols, float *__restrict__ deq, float *__restrict__ ded, float *__restrict__ loss)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= pairs) return;
    const float *a = eq + i * cols, *b = ed + i * cols;
    float s = 0.f;
    for (int j = lane; j < cols; j += 32) s = fmaf(a[j], b[j], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float wi = w ? w[i] : 1.f;
    const float r = s - y[i];
    const float g = 2.f * wi * r / wsum;
    if (lane == 0) atomicAdd(loss, wi * r * r / wsum);
    for (int j = lane; j < cols; j += 32) {
        deq[i * cols + j] = g * b[j];
        ded[i * cols + j] = g * a[j];
    }
}

// dz = (de - e (e . de)) / |z|; one warp per row (in place on de).
__global__ void normalize_backward_kernel(const float *__restrict__ e, const float *__restrict__ norm,
                                          float *__restrict__ de, int64_t rows, int cols)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    const float *er = e + r * cols;
    float *dr = de + r * cols;
    float dot = 0.f;
    for (int j = lane; j < cols; j += 32) dot = fmaf(er[j], dr[j], dot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    const float inv = 1.f / norm[r];
    for (int j = lane; j < cols; j += 32) dr[j] = (dr[j] - er[j] * dot) * inv;
}

// da *= gelu'(h) in place.
__global__ void gelu_backward_kernel(const float *__restrict__ h, float *__restrict__ da, int64_t count)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) da[i] *= gelu_grad(h[i]);
}

// out[j] += sum_r x[r, j]: block (32 columns x 8 row lanes) over a chunk of
// 256 rows, shared-memory reduction, one atomic per column and block.
__global__ void colsum_kernel(const float *__restrict__ x, int64_t rows, int cols, float *__restrict__ out)
{
    __shared__ float part[8][33];
    const int c = blockIdx.x * 32 + (threadIdx.x & 31);
    const int lane_r = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.y * 256;
    float s = 0.f;
    if (c < cols)
        for (int64_t r = r0 + lane_r; r < min(rows, r0 + 256); r += 8) s += x[r * cols + c];
    part[lane_r][threadIdx.x & 31] = s;
    __syncthreads();
    if (lane_r == 0 && c < cols) {
        float t = 0.f;
        for (int i = 0; i < 8; ++i) t += part[i][threadIdx.x & 31];
        atomicAdd(out + c, t);
    }
}

// dst[r, c] = bf16(src[r, c]) for c < cols, 0 for cols <= c < ldd.
__global__ void to_bf16_padded_kernel(const float *__restrict__ src, int64_t rows, int cols, uint16_t *__restrict__ dst,
                                      int ldd)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * ldd) return;
    const int64_t r = i / ldd;
    const int c = (int)(i - r * ldd);
    dst[i] = c < cols ? bf16_bits(src[r * cols + c]) : (uint16_t)0;
}

// ---------------------------------------------------------------------------
// The tensor-core training step's elementwise kernels.  The step is bound by
// the passes over its activations (8,192 stacked rows x 512), so each kernel
// reads its input once and writes every form the contractions need -- the row-
// major BF16 operand and the transposed one (rows as K, zero past the last row
// up to the contraction's padded length) -- from one 32 x 64 tile staged in
// shared memory.
// ---------------------------------------------------------------------------

constexpr int TR = 32, TC = 64;         // rows and columns of a tile
constexpr int TSTRIDE = TC + 2;         // (transposed reads of a column pair stay conflict-free)

// Eight consecutive BF16 values of the tile's row tid / 8 into the tile.
__device__ __forceinline__ void tile_put(uint16_t (*tile)[TSTRIDE], int tid, const uint16_t v[8])
{
    uint32_t *w = reinterpret_cast<uint32_t *>(&tile[tid >> 3][(tid & 7) * 8]);
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = (uint32_t)v[2 * u] | (uint32_t)v[2 * u + 1] << 16;
}

// The tile transposed: dst[c0 + c][r0 .. r0 + 31] (16 bytes per thread; ldd a
// multiple of 8, r0 of 32) for c0 + c < cols.
__device__ __forceinline__ void tile_write_t(const uint16_t (*tile)[TSTRIDE], int tid, uint16_t *__restrict__ dst,
                                             int64_t ldd, int c0, int cols, int64_t r0)
{
    const int c = tid >> 2, k = (tid & 3) * 8;
    if (c0 + c >= cols) return;
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = (uint32_t)tile[k + 2 * u][c] | (uint32_t)tile[k + 2 * u + 1][c] << 16;
    *reinterpret_cast<uint4 *>(dst + (int64_t)(c0 + c) * ldd + r0 + k) = make_uint4(w[0], w[1], w[2], w[3]);
}

// The first row of a block's tile: the tiles of more rows than blockIdx.y may count
// go on in blockIdx.z (a last plane's blocks past the rows have nothing to do).
constexpr unsigned kGridY = 65535;
__device__ __forceinline__ int64_t tile_row0() { return ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * TR; }
dim3 tile_grid(int64_t cols, int64_t rows)
{
    const int64_t t = (rows + TR - 1) / TR;
    return dim3((unsigned)(cols / TC), (unsigned)(t < kGridY ? t : kGridY), (unsigned)((t + kGridY - 1) / kGridY));
}

// The step's stacked input rows (query rows 0 .. b - 1, descriptor rows b ..
// 2b - 1; D_pad long) and their transpose [D, K].  With pairs.row gathered
// (pair k of the order: base[n_scenes] row row[k], and base[scene[k]] row
// obj[k]) and written to x; without read from x.
__global__ void __launch_bounds__(256)
train_rows_kernel(TrainPairs pairs, int64_t off, int64_t b, int D, int D_pad, uint16_t *__restrict__ x,
                  uint16_t *__restrict__ xT, int64_t K)
{
    __shared__ __align__(4) uint16_t tile[TR][TSTRIDE];
    const int tid = threadIdx.x;
    const int c0 = blockIdx.x * TC;
    const int64_t r0 = tile_row0();
    if (r0 >= K) return;
    const int64_t r = r0 + (tid >> 3);
    const int c = c0 + (tid & 7) * 8;           // (D_pad is a multiple of 64: the tile's columns exist)
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r < 2 * b) {
        const uint16_t *src;
        if (pairs.row) {
            const int k = pairs.perm[off + (r < b ? r : r - b)];
            src = r < b ? pairs.base[pairs.n_scenes] + (int64_t)pairs.row[k] * D_pad
                        : pairs.base[pairs.scene ? pairs.scene[k] : 0] + (int64_t)pairs.obj[k] * D_pad;
        } else {
            src = x + r * D_pad;
        }
        v = *reinterpret_cast<const uint4 *>(src + c);
        if (pairs.row) *reinterpret_cast<uint4 *>(x + r * D_pad + c) = v;
    }
    const uint16_t h[8] = {(uint16_t)v.x, (uint16_t)(v.x >> 16), (uint16_t)v.y, (uint16_t)(v.y >> 16),
                           (uint16_t)v.z, (uint16_t)(v.z >> 16), (uint16_t)v.w, (uint16_t)(v.w >> 16)};
    tile_put(tile, tid, h);
    __syncthreads();
    tile_write_t(tile, tid, xT, K, c0, D, r0);
}

// ab = bf16(gelu(h + b)) [rows, cols], and its transpose aT [cols, K]
// (nullable); h is left as the contraction wrote it (the backward pass adds b
// again).  cols a multiple of 64.
__global__ void __launch_bounds__(256)
gelu_bf16_kernel(const float *__restrict__ h, const float *__restrict__ b, int64_t rows, int cols,
                 uint16_t *__restrict__ ab, uint16_t *__restrict__ aT, int64_t K)
{
    __shared__ __align__(4) uint16_t tile[TR][TSTRIDE];
    const int tid = threadIdx.x;
    const int c0 = blockIdx.x * TC;
    const int64_t r0 = tile_row0();
    if (r0 >= (aT ? K : rows)) return;
    const int64_t r = r0 + (tid >> 3);
    const int c = c0 + (tid & 7) * 8;
    uint16_t g[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (r < rows) {
        const float4 *hp = reinterpret_cast<const float4 *>(h + r * cols + c);
        const float4 *bp = reinterpret_cast<const float4 *>(b + c);
        const float4 h0 = hp[0], h1 = hp[1], b0 = __ldg(bp), b1 = __ldg(bp + 1);
        const float v[8] = {h0.x + b0.x, h0.y + b0.y, h0.z + b0.z, h0.w + b0.w,
                            h1.x + b1.x, h1.y + b1.y, h1.z + b1.z, h1.w + b1.w};
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = bf16_bits(gelu(v[u]));
        *reinterpret_cast<uint4 *>(ab + r * cols + c) =
            make_uint4((uint32_t)g[0] | (uint32_t)g[1] << 16, (uint32_t)g[2] | (uint32_t)g[3] << 16,
                       (uint32_t)g[4] | (uint32_t)g[5] << 16, (uint32_t)g[6] | (uint32_t)g[7] << 16);
    }
    if (!aT) return;
    tile_put(tile, tid, g);
    __syncthreads();
    tile_write_t(tile, tid, aT, K, c0, cols, r0);
}

// Both bias gradients are column sums over the stacked rows in one fixed order:
// per GB_ROWS rows eight partial sums of every eighth row in row order, those
// eight in order, then the blocks' sums in order (by the block that comes last
// to its columns).  Summed by one atomic per 32 pairs, b2's gradient differed by
// up to 1.3e-7 between two runs at 1,024 pairs, which flips BF16 roundings of
// the weights: W1 then moved by up to 2e-5 in a run of five steps.  The fixed
// order costs an epoch of 120,000 pairs 2% (5.98 -> 6.11 ms).
constexpr int GB_ROWS = 256, GB_STEP = 64;

// dh = da gelu'(h + b) as its BF16 transpose dhT [cols, K], and its column
// sums gb.  The blocks past the column tiles sum those of dz [rows, P] to gb2.
// Two 32-row tiles per step of 512 threads.  part: gridDim.x * gridDim.y * TC
// floats; done: gridDim.x counts, 0 before and after.
__global__ void __launch_bounds__(512)
gelu_backward_t_kernel(const float *__restrict__ h, const float *__restrict__ b, const float *__restrict__ da,
                       int64_t rows, int cols, uint16_t *__restrict__ dhT, int64_t K, float *__restrict__ gb,
                       const float *__restrict__ dz, int P, float *__restrict__ gb2, float *__restrict__ part,
                       int32_t *__restrict__ done)
{
    __shared__ bool s_last;
    __shared__ __align__(4) uint16_t tile[2][TR][TSTRIDE];
    __shared__ float xs[GB_STEP][TC + 1];
    const int tid = threadIdx.x;
    const int sr = tid >> 6, sc = tid & 63;     // this thread's partial sum: rows sr mod 8, column sc
    const int64_t base = (int64_t)blockIdx.y * GB_ROWS;
    const int tiles = cols / TC;
    float acc = 0.f;
    float *out;
    bool mine;
    if ((int)blockIdx.x < tiles) {
        const int half = tid >> 8, lt = tid & 255;
        const int c0 = blockIdx.x * TC;
        const int c = c0 + (lt & 7) * 8;
        const float4 *bp = reinterpret_cast<const float4 *>(b + c);
        const float4 b0 = __ldg(bp), b1 = __ldg(bp + 1);
        for (int64_t s0 = base; s0 < min(K, base + GB_ROWS); s0 += GB_STEP) {     // (K a multiple of GB_STEP)
            const int row = half * TR + (lt >> 3);
            const int64_t r = s0 + row;
            uint16_t g[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            float x[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (r < rows) {
                const float4 *hp = reinterpret_cast<const float4 *>(h + r * cols + c);
                const float4 *dp = reinterpret_cast<const float4 *>(da + r * cols + c);
                const float4 h0 = hp[0], h1 = hp[1], d0 = dp[0], d1 = dp[1];
                const float v[8] = {h0.x + b0.x, h0.y + b0.y, h0.z + b0.z, h0.w + b0.w,
                                    h1.x + b1.x, h1.y + b1.y, h1.z + b1.z, h1.w + b1.w};
                const float d[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    x[u] = d[u] * gelu_grad(v[u]);
                    g[u] = bf16_bits(x[u]);
                }
            }
            tile_put(tile[half], lt, g);
#pragma unroll
            for (int u = 0; u < 8; ++u) xs[row][(lt & 7) * 8 + u] = x[u];
            __syncthreads();
            tile_write_t(tile[half], lt, dhT, K, c0, cols, s0 + half * TR);
#pragma unroll
            for (int k = 0; k < GB_STEP / 8; ++k) acc += xs[sr + 8 * k][sc];      // (zero past the last row)
            __syncthreads();
        }
        out = gb + c0;
        mine = true;
    } else {
        const int c0 = ((int)blockIdx.x - tiles) * TC;
        mine = c0 + sc < P;
        if (mine)
            for (int64_t r = base + sr; r < min(rows, base + GB_ROWS); r += 8) acc += dz[r * P + c0 + sc];
        out = gb2 + c0;
    }
    xs[sr][sc] = acc;
    __syncthreads();
    if (tid < TC) {
        float t = 0.f;
        for (int i = 0; i < 8; ++i) t += xs[i][tid];
        part[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * TC + tid] = t;
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(done + blockIdx.x, 1) == (int)gridDim.y - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) done[blockIdx.x] = 0;
    if (tid < TC && mine) {
        float t = 0.f;
        for (int y = 0; y < (int)gridDim.y; ++y) t += __ldcg(part + ((int64_t)y * gridDim.x + blockIdx.x) * TC + tid);
        out[tid] = t;
    }
}

// One warp per pair (LP_PAIRS pairs per block): both rows' bias and
// normalisation, the pair's loss, and the gradient back through the
// normalisation, held in registers (NPL values of each row per lane) and
// written as dz FP32 [2b, P] (for the bias sums), BF16 and the transpose dzT
// [P, K] (zero from 2b), with the loss added to *loss.
constexpr int LP_PAIRS = 32;
template <int NPL>
__global__ void __launch_bounds__(256)
pair_step_kernel(const float *__restrict__ z, const float *__restrict__ b2, TrainPairs pairs, int64_t off, float wsum,
                 int64_t b, int P, float *__restrict__ dzf, uint16_t *__restrict__ dzb,
                 uint16_t *__restrict__ dzT, int64_t K, float *__restrict__ loss)
{
    extern __shared__ __align__(16) uint16_t lp_tile[];     // [2][LP_PAIRS][P + 2]
    __shared__ float s_loss[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * LP_PAIRS;
    const int ldt = P + 2;
    const unsigned FULL = 0xffffffffu;
    float lsum = 0.f;
    for (int t = warp; t < LP_PAIRS; t += 8) {
        const int64_t i = i0 + t;
        if (i >= b) break;
        const float *zr[2] = {z + i * P, z + (b + i) * P};
        float e[2][NPL], nrm[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float ss = 0.f;
#pragma unroll
            for (int k = 0; k < NPL; ++k) {
                const int j = lane + 32 * k;
                const float v = j < P ? zr[q][j] + __ldg(b2 + j) : 0.f;
                e[q][k] = v;
                ss = fmaf(v, v, ss);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(FULL, ss, o);
            nrm[q] = fmaxf(sqrtf(ss), 1e-20f);
#pragma unroll
            for (int k = 0; k < NPL; ++k) e[q][k] = e[q][k] / nrm[q];
        }
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < NPL; ++k) s = fmaf(e[0][k], e[1][k], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        const int64_t at = pairs.perm ? pairs.perm[off + i] : off + i;
        const float wi = pairs.w ? pairs.w[at] : 1.f;
        const float r = s - pairs.y[at];
        const float g = 2.f * wi * r / wsum;
        lsum += wi * r * r / wsum;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float dot = 0.f;
#pragma unroll
            for (int k = 0; k < NPL; ++k) dot = fmaf(e[q][k], g * e[1 - q][k], dot);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(FULL, dot, o);
            const float inv = 1.f / nrm[q];
#pragma unroll
            for (int k = 0; k < NPL; ++k) {
                const int j = lane + 32 * k;
                if (j >= P) continue;
                const float dz = fmaf(-e[q][k], dot, __fmul_rn(g, e[1 - q][k])) * inv;
                dzf[(q * b + i) * P + j] = dz;
                const uint16_t h = bf16_bits(dz);
                dzb[(q * b + i) * P + j] = h;
                lp_tile[(q * LP_PAIRS + t) * ldt + j] = h;
            }
        }
    }
    if (lane == 0) s_loss[warp] = lsum;
    __syncthreads();
    // the transposes: a warp per column, its lanes the block's pairs
    const int np = (int)min((int64_t)LP_PAIRS, b - i0);
    for (int p = warp; p < P; p += 8) {
        if (lane < np) {
            dzT[(int64_t)p * K + i0 + lane] = lp_tile[lane * ldt + p];
            dzT[(int64_t)p * K + b + i0 + lane] = lp_tile[(LP_PAIRS + lane) * ldt + p];
        }
    }
    // this block's share of the columns past the last row
    const int64_t pad = K - 2 * b, share = (pad + gridDim.x - 1) / gridDim.x;
    const int64_t z0 = 2 * b + blockIdx.x * share, z1 = min(K, z0 + share);
    for (int p = warp; p < P; p += 8)
        for (int64_t k = z0 + lane; k < z1; k += 32) dzT[(int64_t)p * K + k] = 0;
    // the loss over the block's warps
    if (tid == 0) {
        float t = 0.f;
        for (int v = 0; v < 8; ++v) t += s_loss[v];
        atomicAdd(loss, t);
    }
}

// e = bf16((z + b) / |z + b|), one warp per row (the inference path).
__global__ void normalize_bf16_kernel(const float *__restrict__ z, const float *__restrict__ b, int64_t rows, int cols,
                                      uint16_t *__restrict__ e)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    const float *zr = z + r * cols;
    float ss = 0.f;
    for (int j = lane; j < cols; j += 32) {
        const float v = zr[j] + b[j];
        ss = fmaf(v, v, ss);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float nrm = fmaxf(sqrtf(ss), 1e-20f);
    for (int j = lane; j < cols; j += 32) e[r * cols + j] = bf16_bits((zr[j] + b[j]) / nrm);
}

// The BF16 operand copies of parameter i of [W1 | b1 | W2 | b2]: W1 in w1b
// [H, D_pad] (whose padding stays zero), W2 in w2b [P, H] and transposed in
// w2t [H, P].
__device__ __forceinline__ void store_weight(int64_t i, float v, const MlpShape &m)
{
    const int64_t n1 = (int64_t)m.H * m.D;
    if (i < n1) {
        const int64_t h = i / m.D;
        m.w1b[h * m.D_pad + (i - h * m.D)] = bf16_bits(v);
        return;
    }
    const int64_t j = i - n1 - m.H;
    if (j >= 0 && j < (int64_t)m.P * m.H) {
        const int64_t p = j / m.H;
        const uint16_t x = bf16_bits(v);
        m.w2b[j] = x;
        m.w2t[(j - p * m.H) * m.P + p] = x;
    }
}

__global__ void weights_bf16_kernel(const float *__restrict__ p, int64_t count, MlpShape m)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) store_weight(i, p[i], m);
}

// Adam with bias correction (step t >= 1), then the updated weights' BF16 copies.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int64_t count, float lr, float b1, float b2, float eps, int t,
                            MlpShape shape)
{
    __shared__ float s_c[2];
    if (threadIdx.x < 2) s_c[threadIdx.x] = 1.f - powf(threadIdx.x ? b2 : b1, (float)t);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / s_c[0];
    const float vh = vi / s_c[1];
    const float x = p[i] - lr * mh / (sqrtf(vh) + eps);
    p[i] = x;
    store_weight(i, x, shape);
}

unsigned blocks_for(int64_t n, int th) { return (unsigned)((n + th - 1) / th); }

}  // namespace

cudaError_t mlp_gemm(bool ta, bool tb, int M, int N, int K, float alpha, const float *A, int lda, const float *B,
                     int ldb, float beta, float *C, int ldc, cudaStream_t s)
{
    if (M <= 0 || N <= 0) return cudaSuccess;
    dim3 grid((unsigned)((N + 63) / 64), (unsigned)((M + 63) / 64));
    if (!ta && !tb) gemm_f32_kernel<false, false><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    else if (!ta && tb) gemm_f32_kernel<false, true><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    else if (ta && !tb) gemm_f32_kernel<true, false><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    else gemm_f32_kernel<true, true><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    return cudaGetLastError();
}

cudaError_t mlp_bias_gelu(float *h, const float *b, float *a, int64_t rows, int cols, cudaStream_t s)
{
    if (rows * cols <= 0) return cudaSuccess;
    bias_gelu_kernel<<<blocks_for(rows * cols, 256), 256, 0, s>>>(h, b, a, rows, cols);
    return cudaGetLastError();
}

cudaError_t mlp_to_bf16_padded(const float *src, int64_t rows, int cols, uint16_t *dst, int ldd, cudaStream_t s)
{
    if (rows <= 0 || ldd <= 0) return cudaSuccess;
    if (ldd < cols) return cudaErrorInvalidValue;
    to_bf16_padded_kernel<<<blocks_for(rows * ldd, 256), 256, 0, s>>>(src, rows, cols, dst, ldd);
    return cudaGetLastError();
}

cudaError_t mlp_bias_normalize(float *z, const float *b, float *e, float *norm, int64_t rows, int cols,
                               cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    bias_normalize_kernel<<<blocks_for(rows, 8), 256, 0, s>>>(z, b, e, norm, rows, cols);
    return cudaGetLastError();
}

cudaError_t mlp_pair_loss(const float *eq, const float *ed, const float *y, const float *w, float wsum, int64_t pairs,
                          int cols, float *deq, float *ded, float *loss, cudaStream_t s)
{
    if (pairs <= 0) return cudaSuccess;
    pair_loss_kernel<<<blocks_for(pairs, 8), 256, 0, s>>>(eq, ed, y, w, wsum, pairs, cols, deq, ded, loss);
    return cudaGetLastError();
}

cudaError_t mlp_normalize_backward(const float *e, const float *norm, float *de, int64_t rows, int cols,
                                   cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    normalize_backward_kernel<<<blocks_for(rows, 8), 256, 0, s>>>(e, norm, de, rows, cols);
    return cudaGetLastError();
}

cudaError_t mlp_gelu_backward(const float *h, float *da, int64_t count, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    gelu_backward_kernel<<<blocks_for(count, 256), 256, 0, s>>>(h, da, count);
    return cudaGetLastError();
}

cudaError_t mlp_colsum(const float *x, int64_t rows, int cols, float *out, bool accumulate, cudaStream_t s)
{
    if (cols <= 0) return cudaSuccess;
    if (!accumulate) {
        cudaError_t e = cudaMemsetAsync(out, 0, (size_t)cols * sizeof(float), s);
        if (e != cudaSuccess) return e;
    }
    if (rows <= 0) return cudaSuccess;
    dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 255) / 256));
    colsum_kernel<<<grid, 256, 0, s>>>(x, rows, cols, out);
    return cudaGetLastError();
}

cudaError_t mlp_train_rows(const TrainPairs &pairs, int64_t off, int64_t b, int D, int D_pad, uint16_t *x, uint16_t *xT,
                           int64_t K, cudaStream_t s)
{
    if (b < 1 || D_pad % TC != 0 || K % 64 != 0 || K < 2 * b || (pairs.row && !pairs.perm)) return cudaErrorInvalidValue;
    train_rows_kernel<<<tile_grid(D_pad, K), 256, 0, s>>>(pairs, off, b, D, D_pad, x, xT, K);
    return cudaGetLastError();
}

cudaError_t mlp_gelu_bf16(const float *h, const float *b, int64_t rows, int cols, uint16_t *ab, uint16_t *aT, int64_t K,
                          cudaStream_t s)
{
    if (rows < 1 || cols % TC != 0 || (aT && (K % 64 != 0 || K < rows))) return cudaErrorInvalidValue;
    gelu_bf16_kernel<<<tile_grid(cols, aT ? K : rows), 256, 0, s>>>(h, b, rows, cols, ab, aT, K);
    return cudaGetLastError();
}

cudaError_t mlp_gelu_backward_t(const float *h, const float *b, const float *da, int64_t rows, int cols, uint16_t *dhT,
                                int64_t K, float *gb, const float *dz, int P, float *gb2, float *part, int32_t *done,
                                cudaStream_t s)
{
    if (rows < 1 || P < 1 || cols % TC != 0 || K % GB_STEP != 0 || K < rows) return cudaErrorInvalidValue;
    dim3 grid((unsigned)(cols / TC + (P + TC - 1) / TC), (unsigned)((K + GB_ROWS - 1) / GB_ROWS));
    gelu_backward_t_kernel<<<grid, 512, 0, s>>>(h, b, da, rows, cols, dhT, K, gb, dz, P, gb2, part, done);
    return cudaGetLastError();
}

cudaError_t mlp_pair_step(const float *z, const float *b2, const TrainPairs &pairs, int64_t off, float wsum, int64_t b,
                          int P, float *dzf, uint16_t *dzb, uint16_t *dzT, int64_t K, float *loss, cudaStream_t s)
{
    if (b < 1 || P < 32 || P > 1024 || K < 2 * b) return cudaErrorInvalidValue;
    // the tile, 64 rows of P + 2 values
    const size_t smem = (size_t)2 * LP_PAIRS * (P + 2) * sizeof(uint16_t);
    auto kern = P <= 64 ? pair_step_kernel<2> : P <= 128 ? pair_step_kernel<4> : P <= 256 ? pair_step_kernel<8>
                : P <= 512 ? pair_step_kernel<16> : pair_step_kernel<32>;
    if (smem + 1024 > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<(unsigned)((b + LP_PAIRS - 1) / LP_PAIRS), 256, smem, s>>>(z, b2, pairs, off, wsum, b, P, dzf, dzb, dzT, K,
                                                                     loss);
    return cudaGetLastError();
}

cudaError_t mlp_normalize_bf16(const float *z, const float *b, int64_t rows, int cols, uint16_t *e, cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    normalize_bf16_kernel<<<blocks_for(rows, 8), 256, 0, s>>>(z, b, rows, cols, e);
    return cudaGetLastError();
}

cudaError_t mlp_weights_bf16(const float *p, int64_t count, const MlpShape &m, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(m.w1b, 0, (size_t)m.H * m.D_pad * sizeof(uint16_t), s);
    if (e != cudaSuccess) return e;
    weights_bf16_kernel<<<blocks_for(count, 256), 256, 0, s>>>(p, count, m);
    return cudaGetLastError();
}

cudaError_t mlp_adam(float *p, const float *g, float *m, float *v, int64_t count, float lr, int t, const MlpShape &shape,
                     cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    adam_kernel<<<blocks_for(count, 256), 256, 0, s>>>(p, g, m, v, count, lr, 0.9f, 0.999f, 1e-8f, t, shape);
    return cudaGetLastError();
}

}  // namespace farm
