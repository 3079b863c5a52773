// k_assoc.cu -- mapping-side association of a batch of detections with the
// memory's entities (App. D.1 steps 3-5), each a 3D Gaussian (mean;
// covariance packed xx, xy, xz, yy, yz, zz) with an appearance feature:
//
//  * neighbour search: from the detection-by-entity feature cosines (the
//    FP32-accurate similarity kernel), the active entities with cosine >=
//    tau_f get the Hellinger distance
//      H = sqrt(1 - BC),  ln BC = (ln det S_d + ln det S_e) / 4 - ln det S / 2
//                                 - dmu' S^-1 dmu / 8,  S = (S_d + S_e) / 2,
//    (1 - BC evaluated as -expm1(ln BC)); those with H <= h_max are sorted by
//    (H, index) and the first max_m kept (one CTA per detection).  For
//    enough cosines, of more than kSimFewRows detections, the similarity kernel
//    keeps only those reaching tau_f (the emitting form of the fused rank selection, its
//    threshold tau_f for every row), so the detection-by-entity block is
//    neither written nor read; a detection with more of them than its buffer
//    holds is searched over its stored row, which is then computed;
//  * correspondence: the connected components of the graph joining each
//    detection (node N + d) to its matches: a union-find over smallest nodes
//    (roots hooked by compare-and-swap: every step moves a label to a smaller
//    node, so it ends whatever the order), each detection's matches united as
//    soon as they are found; the winner of a component is its entity of
//    largest weight (lower index on ties), a component without an entity is a
//    lone detection that starts a new entity;
//  * fusion: a warp per slot; a winner sums w (mu - c) and w f over the slots
//    merged into it (listed per winner; c the winner's own mean: a shift that
//    keeps FP32 digits at site coordinates), then w (S + (mu - mu_g)(mu -
//    mu_g)') -- the sufficient-statistics merge M1 = w mu, M2 = w (S + mu mu')
//    in a form free of the cancellation of M2 / w - mu mu'.  The members'
//    order (and the last bits) may vary from run to run.
//
// 4,096 detections x 20,000 entities, F = 256: 183 us a call against 300 when
// the similarity stored the 328 MB block and a scan read it back, the
// components took one CTA's rounds and the fusion four passes of atomics
// (search 106 -> 25 us, components 57 -> the match kernel's tail, fusion and its
// clearing 106 -> 39; the similarity 124 -> 111, 60% of the tensor rate: 17
// tiles of eight K slices per CTA pair, each waiting for its fold).
#include "farm_internal.h"

namespace farm {
namespace {

constexpr int TA = 128;
constexpr int CAPA = 1024;       // candidates within the budget a detection may have
constexpr int CAPP = 4096;       // prefilter list: entities past the cosine threshold awaiting evaluation
constexpr int PER_PASS = TA * 16;   // entries one streaming pass can add (four float4 per thread)

__device__ __forceinline__ float det3f(const float c[6])
{
    return c[0] * (c[3] * c[5] - c[4] * c[4]) - c[1] * (c[1] * c[5] - c[4] * c[2]) +
           c[2] * (c[1] * c[4] - c[3] * c[2]);
}

// Hellinger distance of two Gaussians; 1 for a degenerate covariance.
__device__ float hellinger_f(const float m1[3], const float c1[6], const float m2[3], const float c2[6])
{
    float S[6], d[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) S[k] = 0.5f * (c1[k] + c2[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = m1[k] - m2[k];
    const float dS = det3f(S), d1 = det3f(c1), d2 = det3f(c2);
    if (!(dS > 0.f) || !(d1 > 0.f) || !(d2 > 0.f)) return 1.f;
    const float a0 = S[3] * S[5] - S[4] * S[4], a1 = S[2] * S[4] - S[1] * S[5], a2 = S[1] * S[4] - S[2] * S[3];
    const float a3 = S[0] * S[5] - S[2] * S[2], a4 = S[1] * S[2] - S[0] * S[4], a5 = S[0] * S[3] - S[1] * S[1];
    const float x0 = a0 * d[0] + a1 * d[1] + a2 * d[2];
    const float x1 = a1 * d[0] + a3 * d[1] + a4 * d[2];
    const float x2 = a2 * d[0] + a4 * d[1] + a5 * d[2];
    const float q = (d[0] * x0 + d[1] * x1 + d[2] * x2) / dS;
    const float lbc = 0.25f * (logf(d1) + logf(d2)) - 0.5f * logf(dS) - 0.125f * q;
    return sqrtf(fmaxf(-expm1f(lbc), 0.f));
}

// The Hellinger distance of detection (md, cd) to entity e, -1 for an
// inactive entity.  Kept out of line: the streaming loop that calls it for
// the few entities past the cosine prefilter is unrolled sixteen-fold, and
// inlining it there overflowed the instruction cache.
__device__ __noinline__ float entity_distance(int e, int32_t N, const float *__restrict__ ent_mu,
                                              const float *__restrict__ ent_cov,
                                              const int32_t *__restrict__ ent_active, const float md[3],
                                              const float cd[6])
{
    if (!ent_active[e]) return -1.f;
    float me[3], ce[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) me[k] = ent_mu[(int64_t)k * N + e];
#pragma unroll
    for (int k = 0; k < 6; ++k) ce[k] = ent_cov[(int64_t)k * N + e];
    return hellinger_f(md, cd, me, ce);
}

// The union-find over node labels (label[x] <= x, a root labels itself).  Nodes
// on a walk are pointed at their grandparents; labels are read past L1.
__device__ __forceinline__ int find_root(int32_t *label, int x)
{
    volatile int32_t *l = label;
    int cur = l[x];
    if (cur != x) {
        int prev = x, next;
        while (cur > (next = l[cur])) {
            l[prev] = next;
            prev = cur;
            cur = next;
        }
    }
    return cur;
}

__device__ __forceinline__ void unite(int32_t *label, int u, int v)
{
    int a = find_root(label, u), b = find_root(label, v);
    while (a != b) {
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        // a, the larger root, takes b's label, unless it has been hooked meanwhile
        const int old = atomicCAS(&label[a], a, b);
        if (old == a) break;
        a = find_root(label, old);
    }
}

// The matches of detection d: cnt candidates (H bits, entity) in cand (the
// first CAPA of them), ordered by (H, index), the first max_m written and
// united with the detection's node.  Every thread of the block calls it.
__device__ __forceinline__ void finish_matches(uint64_t *cand, int cnt, int d, int32_t N, int32_t max_m,
                                               int32_t *__restrict__ match_cnt, int32_t *__restrict__ match_idx,
                                               float *__restrict__ match_h, int32_t *label, int32_t *err)
{
    const int tid = threadIdx.x;
    if (cnt > CAPA) {
        if (tid == 0) atomicOr(err, kErrAssocOverflow);
    }
    const int nc = min(cnt, CAPA);
    int P = 1;
    while (P < nc) P <<= 1;
    for (int i = nc + tid; i < P; i += TA) cand[i] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {           // ascending: smaller H, then lower index, first
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < P; i += TA) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const uint64_t a = cand[i], b = cand[ixj];
                    const bool up = (i & k) == 0;
                    if (up ? (a > b) : (a < b)) { cand[i] = b; cand[ixj] = a; }
                }
            }
            __syncthreads();
        }
    }
    if (tid == 0) match_cnt[d] = cnt;
    for (int j = tid; j < max_m; j += TA) {
        const bool has = j < nc;
        const int e = has ? (int)(cand[j] & 0xffffffffu) : -1;
        match_idx[(int64_t)d * max_m + j] = e;
        match_h[(int64_t)d * max_m + j] = has ? __uint_as_float((uint32_t)(cand[j] >> 32)) : -1.f;
        if (has) unite(label, N + d, e);
    }
}

// Before the search: labels, winners and member counts cleared; with the
// emitting similarity, every detection's threshold and an empty buffer.
__global__ void __launch_bounds__(256)
assoc_init_kernel(int32_t T, int32_t B, float tau_f, int32_t *__restrict__ label, unsigned long long *__restrict__ win,
                  int32_t *__restrict__ mcnt, int32_t *__restrict__ counters, uint32_t *__restrict__ tau_key,
                  int32_t *__restrict__ cnt)
{
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t < 2) counters[t] = 0;
    if (t < T) {
        label[t] = t;
        win[t] = 0ull;
        mcnt[t] = 0;
    }
    if (tau_key && t < B) {
        const uint32_t u = __float_as_uint(tau_f + 0.0f);      // the order key of the similarity kernels
        tau_key[t] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
        cnt[t] = 0;
    }
}

// One CTA per detection over the entities its cosine row reached tau_f for
// (buffered by the similarity kernel, in any order); a detection whose buffer
// overflowed is listed for assoc_search_kernel.
__global__ void __launch_bounds__(TA)
assoc_match_kernel(FuseEmit emit, int32_t N, int32_t B, const float *__restrict__ ent_mu,
                   const float *__restrict__ ent_cov, const int32_t *__restrict__ ent_active,
                   const float *__restrict__ det_mu, const float *__restrict__ det_cov, float h_max, int32_t max_m,
                   int32_t *__restrict__ match_cnt, int32_t *__restrict__ match_idx, float *__restrict__ match_h,
                   int32_t *label, int32_t *n_over, int32_t *__restrict__ over, int32_t *err)
{
    __shared__ uint64_t cand[CAPA];
    __shared__ int s_cnt;
    const int d = blockIdx.x, tid = threadIdx.x;
    const int np = emit.cnt[d];
    if (np > emit.cap) {
        if (tid == 0) over[atomicAdd(n_over, 1)] = d;
        return;
    }
    if (tid == 0) s_cnt = 0;
    float md[3], cd[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) md[k] = det_mu[(int64_t)k * B + d];
#pragma unroll
    for (int k = 0; k < 6; ++k) cd[k] = det_cov[(int64_t)k * B + d];
    __syncthreads();
    const uint64_t *words = emit.cand + (int64_t)d * emit.cap;
    for (int i = tid; i < np; i += TA) {
        const int e = (int)(0xffffffffu - (uint32_t)(words[i] & 0xffffffffu));
        const float h = entity_distance(e, N, ent_mu, ent_cov, ent_active, md, cd);
        if (h >= 0.f && h <= h_max) {
            const int pos = atomicAdd(&s_cnt, 1);
            if (pos < CAPA) cand[pos] = ((uint64_t)__float_as_uint(h) << 32) | (uint32_t)e;   // H >= 0: bits order like H
        }
    }
    __syncthreads();
    finish_matches(cand, s_cnt, d, N, max_m, match_cnt, match_idx, match_h, label, err);
}

// Detections over their stored cosine rows: all B of them, or (over non-null)
// the *n_over listed ones.
__global__ void __launch_bounds__(TA)
assoc_search_kernel(const float *__restrict__ S, int64_t ld, int32_t N, int32_t B, const float *__restrict__ ent_mu,
                    const float *__restrict__ ent_cov, const int32_t *__restrict__ ent_active,
                    const float *__restrict__ det_mu, const float *__restrict__ det_cov, float tau_f, float h_max,
                    int32_t max_m, int32_t *__restrict__ match_cnt, int32_t *__restrict__ match_idx,
                    float *__restrict__ match_h, int32_t *label, const int32_t *n_over,
                    const int32_t *__restrict__ over, int32_t *err)
{
    __shared__ uint64_t cand[CAPA];
    __shared__ int32_t pre[CAPP];
    __shared__ int s_cnt, s_np;
    const int tid = threadIdx.x;
    const int count = over ? *n_over : B;
    for (int at = blockIdx.x; at < count; at += gridDim.x) {
        const int d = over ? over[at] : at;
        if (tid == 0) {
            s_cnt = 0;
            s_np = 0;
        }
        __syncthreads();
        float md[3], cd[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) md[k] = det_mu[(int64_t)k * B + d];
#pragma unroll
        for (int k = 0; k < 6; ++k) cd[k] = det_cov[(int64_t)k * B + d];
        // the row is streamed in float4 loads, four in flight per thread (its
        // leading dimension is a multiple of 32 floats, so the row is 16-byte
        // aligned and a load never leaves it); the entities past the cosine
        // prefilter are listed in shared memory and evaluated by all threads
        // together (one entity per thread), whenever the list could overflow in
        // the next pass and at the end: evaluated where they are found, they
        // would each run on one lane of a warp
        const float *row = S + (int64_t)d * ld;
        const float4 *row4 = reinterpret_cast<const float4 *>(row);
        const int n4 = (N + 3) >> 2;
        auto evaluate = [&](int np) {
            for (int i = tid; i < np; i += TA) {
                const int e = pre[i];
                const float h = entity_distance(e, N, ent_mu, ent_cov, ent_active, md, cd);
                if (h >= 0.f && h <= h_max) {
                    const int pos = atomicAdd(&s_cnt, 1);
                    if (pos < CAPA) cand[pos] = ((uint64_t)__float_as_uint(h) << 32) | (uint32_t)e;   // H >= 0: bits order like H
                }
            }
        };
        for (int g0 = 0; g0 < n4; g0 += TA * 4) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int g = g0 + u * TA + tid;
                v[u] = g < n4 ? __ldcs(row4 + g) : make_float4(-2.f, -2.f, -2.f, -2.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e0 = 4 * (g0 + u * TA + tid);
                const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (x[c] >= tau_f && e0 + c < N) pre[atomicAdd(&s_np, 1)] = e0 + c;
            }
            __syncthreads();
            const int np = s_np;
            if (np > CAPP - PER_PASS) {      // (uniform) at most PER_PASS more could come in the next pass
                evaluate(np);
                __syncthreads();
                if (tid == 0) s_np = 0;
                __syncthreads();
            }
        }
        evaluate(s_np);
        __syncthreads();
        finish_matches(cand, s_cnt, d, N, max_m, match_cnt, match_idx, match_h, label, err);
        __syncthreads();          // the next detection reuses the shared arrays
    }
}

// root[t]: its component's smallest node; win[r]: the heaviest entity of
// component r as (w bits, ~index).  (Every union is done: the labels are only
// read.)
__global__ void assoc_winner_kernel(int32_t N, int32_t T, const float *__restrict__ ent_w,
                                    const int32_t *__restrict__ label, int32_t *__restrict__ root,
                                    unsigned long long *win)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int r = label[t];
    for (int up = label[r]; up != r; up = label[r]) r = up;
    root[t] = r;
    if (t >= N) return;
    const unsigned long long k = ((unsigned long long)__float_as_uint(fmaxf(ent_w[t], 0.f)) << 32) |
                                 (unsigned long long)(0xffffffffu - (uint32_t)t);
    atomicMax(&win[r], k);
}

// The winner each slot merges into, and the slot's place among its members.
__global__ void assoc_parent_kernel(int32_t T, const int32_t *__restrict__ root,
                                    const unsigned long long *__restrict__ win, int32_t *__restrict__ parent,
                                    int32_t *__restrict__ mcnt, int32_t *__restrict__ pos)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const unsigned long long k = win[root[t]];
    const int p = k ? (int)(0xffffffffu - (uint32_t)(k & 0xffffffffu)) : t;
    parent[t] = p;
    if (p != t) pos[t] = atomicAdd(&mcnt[p], 1);
}

// Each winner's stretch of the members' array (their order is free).
__global__ void assoc_offset_kernel(int32_t T, const int32_t *__restrict__ mcnt, int32_t *__restrict__ off,
                                    int32_t *bump)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < T && mcnt[t] > 0) off[t] = atomicAdd(bump, mcnt[t]);
}

__global__ void assoc_members_kernel(int32_t T, const int32_t *__restrict__ parent, const int32_t *__restrict__ off,
                                     const int32_t *__restrict__ pos, int32_t *__restrict__ members)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int p = parent[t];
    if (p != t) members[off[p] + pos[t]] = t;
}

struct Slots {
    int32_t N, B, F;
    const float *ent_mu, *ent_cov, *ent_feat, *ent_w, *det_mu, *det_cov, *det_feat;
    __device__ float mu(int t, int k) const { return t < N ? ent_mu[(int64_t)k * N + t] : det_mu[(int64_t)k * B + (t - N)]; }
    __device__ float cv(int t, int k) const { return t < N ? ent_cov[(int64_t)k * N + t] : det_cov[(int64_t)k * B + (t - N)]; }
    __device__ const float *feat(int t) const
    {
        return t < N ? ent_feat + (int64_t)t * F : det_feat + (int64_t)(t - N) * F;
    }
    __device__ float w(int t) const { return t < N ? ent_w[t] : 1.f; }
};

constexpr int FW = 8;              // slots (warps) per block of the fusion
constexpr int BIG_MEMBERS = 64;    // a winner of more is fused by its whole block
constexpr int FCHUNK = 512;        // features of a big winner at a time

// out_w, out_mu, out_cov and out_feat of every slot: zeros for a merged one,
// the slot's own values for a winner without members, sums over the members
// (listed at members + off) otherwise.
__global__ void __launch_bounds__(FW * 32)
assoc_fuse_kernel(Slots sl, const int32_t *__restrict__ parent, const int32_t *__restrict__ mcnt,
                  const int32_t *__restrict__ off, const int32_t *__restrict__ members, float *__restrict__ out_w,
                  float *__restrict__ out_mu, float *__restrict__ out_cov, float *__restrict__ out_feat, int vec)
{
    __shared__ float s_part[FW][FCHUNK];
    __shared__ float s_sum[FW][4], s_cov[FW][6], s_mean[4];
    const int T = sl.N + sl.B, F = sl.F;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    const int t0 = blockIdx.x * FW, t = t0 + warp;
    const unsigned FULL = 0xffffffffu;
    if (t < T) {
        // (the slot's first features are in flight while the rest is looked up)
        const float4 *ft4 = reinterpret_cast<const float4 *>(sl.feat(t));
        const int nf4 = vec ? F / 4 : 0;
        float4 pre[2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
            pre[u] = lane + 32 * u < nf4 ? __ldg(ft4 + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
        const int m = parent[t] == t ? mcnt[t] : -1;      // -1: merged away
        float *of = out_feat + (int64_t)t * F;
        if (m >= 0 && m <= BIG_MEMBERS) {
            const int32_t *mem = members + (m > 0 ? off[t] : 0);
            // weight, and mean relative to the winner's own (lanes 0-2)
            float W = sl.w(t), dm = 0.f;
            const float mt = lane < 3 ? sl.mu(t, lane) : 0.f;
            for (int k = 0; k < m; ++k) {
                const int s = mem[k];
                const float w = sl.w(s);
                W += w;
                if (lane < 3) dm += w * (sl.mu(s, lane) - mt);
            }
            const bool own = W > 0.f;
            const float mean = own ? mt + dm / W : 0.f;
            if (lane == 0) out_w[t] = own ? W : 0.f;
            if (lane < 3) out_mu[(int64_t)lane * T + t] = mean;
            // covariance about the fused mean (lanes 0-5)
            const int c = lane < 6 ? lane : 0, a = ia[c], b = ib[c];
            const float ma = __shfl_sync(FULL, mean, a), mb = __shfl_sync(FULL, mean, b);
            if (lane < 6) {
                float acc = sl.w(t) * (sl.cv(t, c) + (sl.mu(t, a) - ma) * (sl.mu(t, b) - mb));
                for (int k = 0; k < m; ++k) {
                    const int s = mem[k];
                    acc += sl.w(s) * (sl.cv(s, c) + (sl.mu(s, a) - ma) * (sl.mu(s, b) - mb));
                }
                out_cov[(int64_t)c * T + t] = own ? acc / W : 0.f;
            }
            // features
            const float wt = sl.w(t);
            if (vec) {
                for (int j = lane; j < nf4; j += 32) {
                    float4 x = j < 32 ? pre[0] : j < 64 ? pre[1] : __ldg(ft4 + j);
                    x.x *= wt; x.y *= wt; x.z *= wt; x.w *= wt;
                    for (int k = 0; k < m; ++k) {
                        const int s = mem[k];
                        const float w = sl.w(s);
                        const float4 y = __ldg(reinterpret_cast<const float4 *>(sl.feat(s)) + j);
                        x.x = fmaf(w, y.x, x.x); x.y = fmaf(w, y.y, x.y);
                        x.z = fmaf(w, y.z, x.z); x.w = fmaf(w, y.w, x.w);
                    }
                    if (own) { x.x /= W; x.y /= W; x.z /= W; x.w /= W; }
                    else x = make_float4(0.f, 0.f, 0.f, 0.f);
                    reinterpret_cast<float4 *>(of)[j] = x;
                }
            } else {
                const float *ft = sl.feat(t);
                for (int j = lane; j < F; j += 32) {
                    float x = wt * ft[j];
                    for (int k = 0; k < m; ++k) {
                        const int s = mem[k];
                        x = fmaf(sl.w(s), sl.feat(s)[j], x);
                    }
                    of[j] = own ? x / W : 0.f;
                }
            }
        } else if (m < 0) {
            if (lane == 0) out_w[t] = 0.f;
            if (lane < 3) out_mu[(int64_t)lane * T + t] = 0.f;
            if (lane < 6) out_cov[(int64_t)lane * T + t] = 0.f;
            if (vec) {
                for (int j = lane; j < nf4; j += 32)
                    reinterpret_cast<float4 *>(of)[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                for (int j = lane; j < F; j += 32) of[j] = 0.f;
            }
        }
    }
    // winners of many members: the block's warps take every FW-th of them
    for (int q = 0; q < FW; ++q) {
        const int g = t0 + q;
        if (g >= T || parent[g] != g || mcnt[g] <= BIG_MEMBERS) continue;     // (uniform across the block)
        const int m = mcnt[g];
        const int32_t *mem = members + off[g];
        float W = warp == 0 ? sl.w(g) : 0.f, dm = 0.f;
        const float mt = lane < 3 ? sl.mu(g, lane) : 0.f;
        for (int k = warp; k < m; k += FW) {
            const int s = mem[k];
            const float w = sl.w(s);
            W += w;
            if (lane < 3) dm += w * (sl.mu(s, lane) - mt);
        }
        if (lane < 3) s_sum[warp][lane] = dm;
        if (lane == 3) s_sum[warp][3] = W;
        __syncthreads();
        if (warp == 0 && lane < 4) {
            float x = 0.f;
            for (int v = 0; v < FW; ++v) x += s_sum[v][lane];
            s_mean[lane] = x;
        }
        __syncthreads();
        W = s_mean[3];
        const bool own = W > 0.f;
        const int c = lane < 6 ? lane : 0, a = ia[c], b = ib[c];
        const float ma = sl.mu(g, a) + s_mean[a] / W, mb = sl.mu(g, b) + s_mean[b] / W;
        if (lane < 6) {
            float acc = warp == 0 ? sl.w(g) * (sl.cv(g, c) + (sl.mu(g, a) - ma) * (sl.mu(g, b) - mb)) : 0.f;
            for (int k = warp; k < m; k += FW) {
                const int s = mem[k];
                acc += sl.w(s) * (sl.cv(s, c) + (sl.mu(s, a) - ma) * (sl.mu(s, b) - mb));
            }
            s_cov[warp][c] = acc;
        }
        __syncthreads();
        if (warp == 0) {
            if (lane == 0) out_w[g] = own ? W : 0.f;
            if (lane < 3) out_mu[(int64_t)lane * T + g] = own ? mt + s_mean[lane] / W : 0.f;
            if (lane < 6) {
                float x = 0.f;
                for (int v = 0; v < FW; ++v) x += s_cov[v][lane];
                out_cov[(int64_t)lane * T + g] = own ? x / W : 0.f;
            }
        }
        for (int f0 = 0; f0 < F; f0 += FCHUNK) {
            const int fn = min(FCHUNK, F - f0);
            float acc[FCHUNK / 32];
#pragma unroll
            for (int u = 0; u < FCHUNK / 32; ++u) {
                const int j = lane + 32 * u;
                acc[u] = warp == 0 && j < fn ? sl.w(g) * sl.feat(g)[f0 + j] : 0.f;
            }
            for (int k = warp; k < m; k += FW) {
                const int s = mem[k];
                const float w = sl.w(s);
                const float *fs = sl.feat(s) + f0;
#pragma unroll
                for (int u = 0; u < FCHUNK / 32; ++u) {
                    const int j = lane + 32 * u;
                    if (j < fn) acc[u] = fmaf(w, __ldg(fs + j), acc[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < FCHUNK / 32; ++u) s_part[warp][lane + 32 * u] = acc[u];
            __syncthreads();
            for (int j = threadIdx.x; j < fn; j += FW * 32) {
                float x = 0.f;
                for (int v = 0; v < FW; ++v) x += s_part[v][j];
                out_feat[(int64_t)g * F + f0 + j] = own ? x / W : 0.f;
            }
            __syncthreads();
        }
    }
}

}  // namespace

cudaError_t launch_assoc_init(const AssocArgs &a, cudaStream_t s)
{
    const int32_t T = a.N + a.B;
    assoc_init_kernel<<<(unsigned)((T + 255) / 256), 256, 0, s>>>(T, a.B, a.tau_f, a.label, a.win, a.mcnt, a.counters,
                                                                   a.emit.tau_key, a.emit.cnt);
    return cudaGetLastError();
}

cudaError_t launch_assoc_match(const AssocArgs &a, cudaStream_t s)
{
    assoc_match_kernel<<<(unsigned)a.B, TA, 0, s>>>(a.emit, a.N, a.B, a.ent_mu, a.ent_cov, a.ent_active, a.det_mu,
                                                    a.det_cov, a.h_max, a.max_m, a.match_cnt, a.match_idx, a.match_h,
                                                    a.label, a.counters + 1, a.over, a.err);
    return cudaGetLastError();
}

cudaError_t launch_assoc(const AssocArgs &a, cudaStream_t s)
{
    const int32_t N = a.N, B = a.B, T = a.N + a.B;
    if (B < 1 || N < 0 || a.F < 1 || a.max_m < 1 || (int64_t)B * a.max_m > 0x7fffffff) return cudaErrorInvalidValue;
    cudaError_t e;
    // the stored rows: all of them, or those the emitted lists overflowed for
    const int32_t *over = a.emit.cnt ? a.over : nullptr;
    const unsigned grid = over ? (unsigned)(B < 304 ? B : 304) : (unsigned)B;
    assoc_search_kernel<<<grid, TA, 0, s>>>(a.S, a.ld, N, B, a.ent_mu, a.ent_cov, a.ent_active, a.det_mu, a.det_cov,
                                            a.tau_f, a.h_max, a.max_m, a.match_cnt, a.match_idx, a.match_h, a.label,
                                            a.counters + 1, over, a.err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned nb = (unsigned)((T + 255) / 256);
    assoc_winner_kernel<<<nb, 256, 0, s>>>(N, T, a.ent_w, a.label, a.members, a.win);    // (roots: before the members)
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_parent_kernel<<<nb, 256, 0, s>>>(T, a.members, a.win, a.parent, a.mcnt, a.pos);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_offset_kernel<<<nb, 256, 0, s>>>(T, a.mcnt, a.off, a.counters);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_members_kernel<<<nb, 256, 0, s>>>(T, a.parent, a.off, a.pos, a.members);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const Slots sl{N, B, a.F, a.ent_mu, a.ent_cov, a.ent_feat, a.ent_w, a.det_mu, a.det_cov, a.det_feat};
    const uintptr_t al = (uintptr_t)a.ent_feat | (uintptr_t)a.det_feat | (uintptr_t)a.out_feat;
    const int vec = a.F % 4 == 0 && (al & 15u) == 0 ? 1 : 0;
    assoc_fuse_kernel<<<(unsigned)((T + FW - 1) / FW), FW * 32, 0, s>>>(sl, a.parent, a.mcnt, a.off, a.members, a.out_w,
                                                                        a.out_mu, a.out_cov, a.out_feat, vec);
    return cudaGetLastError();
}

}  // namespace farm
