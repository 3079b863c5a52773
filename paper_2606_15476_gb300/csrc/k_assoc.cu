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
//    neither written nor read; the detections with more of them than their
//    buffers hold are gathered, and those rows computed again, stored and
//    searched (every row is, without lists, when a sample of the cosines says
//    that most would overflow);
//  * correspondence: the connected components of the graph joining each
//    detection (node N + d) to its matches: a union-find over smallest nodes
//    (roots hooked by compare-and-swap: every step moves a label to a smaller
//    node, so it ends whatever the order), each detection's matches united as
//    soon as they are found; the winner of a component is its entity of
//    largest weight (lower index on ties), a component without an entity is a
//    lone detection that starts a new entity;
//  * fusion: a warp per slot (blocks for the winners of more than BIG_MEMBERS
//    members, a segment of them at a time); a winner sums w (mu - c) and w f over the slots
//    merged into it (listed per winner; c the winner's own mean: a shift that
//    keeps FP32 digits at site coordinates), then w (S + (mu - mu_g)(mu -
//    mu_g)') -- the sufficient-statistics merge M1 = w mu, M2 = w (S + mu mu')
//    in a form free of the cancellation of M2 / w - mu mu'.  The members'
//    order (and the last bits) may vary from run to run.
//
// 4,096 detections x 20,000 entities, F = 256: 176 us a call against 300 when
// the similarity stored the 328 MB block and a scan read it back, the
// components took one CTA's rounds and the fusion four passes of atomics
// (search 106 -> 25 us, components 57 -> the match kernel's tail, fusion and its
// clearing 106 -> 42; the similarity 124 -> 111, 60% of the tensor rate: 17
// tiles of eight K slices per CTA pair, each waiting for its fold).
#include <cuda_fp16.h>

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

// The union-find over node labels: label[x] <= x, and a root labels itself, so a
// label other than the node's own is always of an ancestor with a smaller
// number.  The walk to the root shortens its path as it goes, by halving
// (Tarjan and van Leeuwen, J. ACM 31, 1984; used on GPUs as intermediate pointer
// jumping by Jaiganesh and Burtscher, HPDC 2018): a node is given its
// grandparent and the walk goes on there.  Walks run against one another and
// against the hooking of roots: whatever label a plain store leaves in a node that
// is no root is an ancestor's, and a root is changed by compare-and-swap only.
// Labels are read past L1.
__device__ __forceinline__ int find_root(int32_t *label, int x)
{
    volatile int32_t *const up = label;
    for (;;) {
        const int parent = up[x];
        if (parent == x) return x;
        const int grand = up[parent];
        if (grand == parent) return parent;
        up[x] = grand;
        x = grand;
    }
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

constexpr int PROBE_BLOCKS = 64, PROBE_PAIRS = 2;      // of them, and cosines a warp samples

// Before the search: labels, winners and member counts cleared; with the
// emitting similarity, every detection's threshold and an empty buffer, and
// whether to emit at all.  A list that overflows costs a second product of its
// row, and appending most of a row costs more than storing it, so 1,024 cosines
// of detections and entities spread over both (the FP16 parts' leading ones) are
// compared with tau_f, and with so many of them above it that the mean list would
// fill more than 7/8 of a buffer every row is stored (the last of the sampling
// warps decides).  4,096 x 20,000, F = 256: 3,000 of the entities alike 324 us
// (320 with every row stored; where all lists fit 209 and 288), classes of 2,222
// 580 (559), all of one class 1,134 (1,101); without the sample, and a second
// product of every row once a list overflows, 454, 1,070 and 2,490.
__global__ void __launch_bounds__(256)
assoc_init_kernel(int32_t T, int32_t N, int32_t B, float tau_f, int32_t *__restrict__ label,
                  unsigned long long *__restrict__ win, int32_t *__restrict__ mcnt, int32_t *__restrict__ counters,
                  uint32_t *__restrict__ tau_key, int32_t *__restrict__ cnt, int32_t cap,
                  const uint16_t *__restrict__ dhi, const uint16_t *__restrict__ ehi, int32_t F_pad, int32_t *probe)
{
    const int tid = threadIdx.x, t = blockIdx.x * 256 + tid;
    if (t < kAssocListRows) counters[t] = 0;
    if (t < T) {
        label[t] = t;
        win[t] = 0ull;
        mcnt[t] = 0;
    }
    if (!tau_key) return;
    if (t < B) {
        const uint32_t u = __float_as_uint(tau_f + 0.0f);      // the order key of the similarity kernels
        tau_key[t] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
        cnt[t] = 0;
    }
    const int blocks = min((int)gridDim.x, PROBE_BLOCKS);
    if ((int)blockIdx.x >= blocks) return;
    const int lane = tid & 31, pairs = blocks * 8 * PROBE_PAIRS, p0 = (blockIdx.x * 8 + (tid >> 5)) * PROBE_PAIRS;
    const uint4 *x[PROBE_PAIRS], *y[PROBE_PAIRS];
    float dot[PROBE_PAIRS];
#pragma unroll
    for (int k = 0; k < PROBE_PAIRS; ++k) {
        const uint32_t p = (uint32_t)(p0 + k);
        // (multiplicative hashing, two constants: places spread evenly over each)
        const int64_t d = __umulhi(p * 2246822519u, (uint32_t)B), e = __umulhi(p * 2654435761u, (uint32_t)N);
        x[k] = reinterpret_cast<const uint4 *>(dhi + d * F_pad);
        y[k] = reinterpret_cast<const uint4 *>(ehi + e * F_pad);
        dot[k] = 0.f;
    }
#pragma unroll 4
    for (int j = lane; j < F_pad / 8; j += 32) {
#pragma unroll
        for (int k = 0; k < PROBE_PAIRS; ++k) {
            const uint4 u = __ldg(x[k] + j), v = __ldg(y[k] + j);
            const uint32_t ua[4] = {u.x, u.y, u.z, u.w}, va[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&ua[i]));
                const float2 g = __half22float2(*reinterpret_cast<const __half2 *>(&va[i]));
                dot[k] = fmaf(f.x, g.x, fmaf(f.y, g.y, dot[k]));
            }
        }
    }
    int hits = 0;
#pragma unroll
    for (int k = 0; k < PROBE_PAIRS; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot[k] += __shfl_xor_sync(0xffffffffu, dot[k], o);
        hits += dot[k] >= tau_f ? 1 : 0;
    }
    // (one word counts the warps and their hits)
    if (lane == 0) {
        const int old = atomicAdd(probe, (1 << 16) | hits);
        if (old >> 16 == blocks * 8 - 1) {
            const int64_t all = (old & 0xffff) + hits;
            atomicExch(probe, 0);
            counters[kAssocListRows] = all * N * 8 <= (int64_t)pairs * cap * 7 ? B : 0;
        }
    }
}

// The unit features' FP16 parts, and the place for those of listed detections.
struct OverRows {
    const uint16_t *dhi, *dlo;
    uint16_t *chi, *clo;
    int32_t F_pad;
};

// Row d's to row k, by the block (out of line: few detections take it).
__device__ __noinline__ void copy_operands(const OverRows o, int d, int k)
{
    const int64_t from = (int64_t)d * o.F_pad, to = (int64_t)k * o.F_pad;
    for (int j = 8 * threadIdx.x; j < o.F_pad; j += 8 * TA) {
        *reinterpret_cast<uint4 *>(o.chi + to + j) = __ldg(reinterpret_cast<const uint4 *>(o.dhi + from + j));
        *reinterpret_cast<uint4 *>(o.clo + to + j) = __ldg(reinterpret_cast<const uint4 *>(o.dlo + from + j));
    }
}

// One CTA per detection over the entities its cosine row reached tau_f for
// (buffered by the similarity kernel, in any order); a detection whose buffer
// overflowed (every one's, when nothing was emitted) is listed for
// assoc_search_kernel, and its unit feature copied to the next row of those that
// the storing similarity multiplies.
__global__ void __launch_bounds__(TA, 12)
assoc_match_kernel(FuseEmit emit, int32_t N, int32_t B, const float *__restrict__ ent_mu,
                   const float *__restrict__ ent_cov, const int32_t *__restrict__ ent_active,
                   const float *__restrict__ det_mu, const float *__restrict__ det_cov, float h_max, int32_t max_m,
                   int32_t *__restrict__ match_cnt, int32_t *__restrict__ match_idx, float *__restrict__ match_h,
                   int32_t *label, int32_t *n_over, int32_t *__restrict__ over, const OverRows rows, int32_t *err)
{
    __shared__ uint64_t cand[CAPA];
    __shared__ int s_cnt;
    const int d = blockIdx.x, tid = threadIdx.x;
    const int np = emit.cnt[d];
    if (np > emit.cap) {
        if (tid == 0) {
            s_cnt = atomicAdd(n_over, 1);
            over[s_cnt] = d;
        }
        __syncthreads();
        copy_operands(rows, d, s_cnt);
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
// the *n_over listed ones, the k-th of whose rows is S's k-th.
__global__ void __launch_bounds__(TA)
assoc_search_kernel(const float *__restrict__ S, int64_t ld, int32_t N, int32_t B, const float *__restrict__ ent_mu,
                    const float *__restrict__ ent_cov, const int32_t *__restrict__ ent_active,
                    const float *__restrict__ det_mu, const float *__restrict__ det_cov, float tau_f, float h_max,
                    int32_t max_m, int32_t *__restrict__ match_cnt, int32_t *__restrict__ match_idx,
                    float *__restrict__ match_h, int32_t *label, const int32_t *n_over,
                    const int32_t *__restrict__ over, int32_t *ticket, int32_t *err)
{
    __shared__ uint64_t cand[CAPA];
    __shared__ int32_t pre[CAPP];
    __shared__ int s_cnt, s_np[3], s_at;
    const int tid = threadIdx.x;
    // (one by one from `ticket` where the grid is smaller than their number may be)
    const int count = over ? *n_over : B;
    if (count == 0) return;
    for (;;) {
        if (tid == 0) {
            s_cnt = 0;
            s_np[0] = s_np[1] = s_np[2] = 0;
            s_at = over ? atomicAdd(ticket, 1) : (int)blockIdx.x;
        }
        __syncthreads();
        const int at = s_at;
        if (at >= count) return;
        const int d = over ? over[at] : at;
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
        const float *row = S + (int64_t)at * ld;
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
        // (a pass counts its entities past the `base` before it in a counter of its
        // own: warps that are ahead fill the next pass's while others read this one's)
        int base = 0, pass = 0;
        for (int g0 = 0; g0 < n4; g0 += TA * 4, pass = pass == 2 ? 0 : pass + 1) {
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
                    if (x[c] >= tau_f && e0 + c < N) pre[base + atomicAdd(&s_np[pass], 1)] = e0 + c;
            }
            __syncthreads();
            base += s_np[pass];
            // (the previous pass's counter, read before this pass's barrier, is filled again in two passes)
            if (tid == 0) s_np[pass == 0 ? 2 : pass - 1] = 0;
            if (base > CAPP - PER_PASS) {    // (uniform) at most PER_PASS more could come in the next pass
                evaluate(base);
                __syncthreads();
                base = 0;
            }
        }
        evaluate(base);
        __syncthreads();
        finish_matches(cand, s_cnt, d, N, max_m, match_cnt, match_idx, match_h, label, err);
        if (!over) return;
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

constexpr int BIG_MEMBERS = 64;    // a winner of more is fused by whole blocks
constexpr int SEG = 1024;          // members of it that a block sums at a time

// Each winner's stretch of the members' array (their order is free), and the
// segments of a winner of many members: (winner, segment) work items, as many
// as bump[kAssocItems] counts in the end.  A winner's place among another's
// members is unused: it counts the winner's finished segments.
__global__ void assoc_offset_kernel(int32_t T, const int32_t *__restrict__ mcnt, int32_t *__restrict__ off,
                                    int32_t *__restrict__ pos, int32_t *bump, int2 *__restrict__ items)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int m = mcnt[t];
    if (m <= 0) return;
    off[t] = atomicAdd(bump, m);
    if (m <= BIG_MEMBERS) return;
    const int segs = (m + SEG - 1) / SEG, at = atomicAdd(bump + kAssocItems, segs);
    pos[t] = 0;
    for (int k = 0; k < segs; ++k) items[at + k] = make_int2(t, k);
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
constexpr int FTH = FW * 32;
constexpr int FU = 3;              // members whose features a lane has in flight
constexpr int BIG_BLOCKS = 304;    // blocks that take the big winners' work items

// The sum over the block's threads of N values each, to every thread.
template <int N>
__device__ __forceinline__ void block_sum(float (&v)[N], float (*part)[8], int lane, int warp)
{
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    __syncthreads();                    // (part is free)
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) part[warp][i] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = 0.f;
#pragma unroll
        for (int w = 0; w < FW; ++w) v[i] += part[w][i];
    }
}

// The members' weighted feature sums of a segment (ids and weights in shared
// memory, n of them, the winner itself counted as one), V floats per lane and
// load: put(j, x) for every feature j.  The lanes share out the columns of a
// stretch of up to 32 loads and, when those are fewer than half a warp, several
// members; eight members' loads are in flight per lane.
template <int V, class Put>
__device__ __forceinline__ void segment_features(const Slots &sl, const int32_t *ids, const float *ws, int n,
                                                 float (*part)[V], int lane, int warp, Put put)
{
    const int cols = sl.F / V;
    for (int c0 = 0; c0 < cols; c0 += 32) {
        const int C = min(32, cols - c0), SUB = 32 / C, sub = lane / C, col = lane - sub * C;
        const bool on = sub < SUB;
        float acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.f;
        for (int k0 = warp * SUB; k0 < n; k0 += FU * FW * SUB) {
            float x[FU][V], w[FU];
#pragma unroll
            for (int u = 0; u < FU; ++u) {
                const int k = k0 + u * FW * SUB + sub;
                const bool in = on && k < n;
                w[u] = in ? ws[k] : 0.f;
                const float *f = in ? sl.feat(ids[k]) + (int64_t)(c0 + col) * V : nullptr;
                if constexpr (V == 4) {
                    const float4 y = in ? __ldg(reinterpret_cast<const float4 *>(f)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    x[u][0] = y.x; x[u][1] = y.y; x[u][2] = y.z; x[u][3] = y.w;
                } else {
                    x[u][0] = in ? __ldg(f) : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < FU; ++u)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = fmaf(w[u], x[u][v], acc[v]);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) part[warp * 32 + lane][v] = acc[v];
        __syncthreads();
        if (threadIdx.x < C * V) {
            const int c = threadIdx.x / V, v = threadIdx.x - c * V;
            float x = 0.f;
            for (int q = 0; q < FW; ++q)
                for (int h = 0; h < SUB; ++h) x += part[q * 32 + h * C + c][v];
            put((c0 + c) * V + v, x);
        }
        __syncthreads();
    }
}

// One segment of a winner of many members: its sums of w, w (mu - c) (c the
// winner's own mean) and w f go to the outputs when it is the winner's only
// one, else to sums (4 + F floats per work item, the winner's from `first` on);
// the block that finishes the winner's last segment adds them in order, and
// sums the covariance about the fused mean over all members.
__device__ __forceinline__ void fuse_big(const Slots &sl, int g, int seg, int item, const int32_t *__restrict__ mem,
                                         int m, int32_t *done, float *sums, int vec, float *__restrict__ out_w,
                                         float *__restrict__ out_mu, float *__restrict__ out_cov,
                                         float *__restrict__ out_feat)
{
    __shared__ int32_t ids[SEG + 1];
    __shared__ float ws[SEG + 1];
    __shared__ __align__(16) float s_part[FTH][4];
    __shared__ float s_red[FW][8];
    __shared__ int s_last;
    const int T = sl.N + sl.B, F = sl.F, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int segs = (m + SEG - 1) / SEG, first = item - seg;
    const int k0 = seg * SEG, n0 = min(SEG, m - k0);
    const float mg[3] = {sl.mu(g, 0), sl.mu(g, 1), sl.mu(g, 2)};
    float a[4] = {0.f, 0.f, 0.f, 0.f};         // w (mu - c), w
#pragma unroll
    for (int u = 0; u < SEG / FTH; ++u) {
        const int k = tid + u * FTH;
        if (k >= n0) continue;
        const int s = mem[k0 + k];
        const float w = sl.w(s);
        ids[k] = s;
        ws[k] = w;
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c] += w * (sl.mu(s, c) - mg[c]);
        a[3] += w;
    }
    int n = n0;
    if (seg == 0) {                            // the winner itself
        if (tid == 0) {
            ids[n0] = g;
            ws[n0] = sl.w(g);
            a[3] += ws[n0];
        }
        ++n;
    }
    block_sum<4>(a, s_red, lane, warp);        // (its barriers also cover ids and ws)
    float *mine = sums + (int64_t)item * (4 + F);
    const bool one = segs == 1;
    {
        const bool own = a[3] > 0.f;
        float *of = one ? out_feat + (int64_t)g * F : mine + 4;
        auto put = [&](int j, float x) { of[j] = one ? (own ? x / a[3] : 0.f) : x; };
        if (vec) segment_features<4>(sl, ids, ws, n, s_part, lane, warp, put);
        else segment_features<1>(sl, ids, ws, n, reinterpret_cast<float(*)[1]>(&s_part[0][0]), lane, warp, put);
    }
    if (!one) {
        if (tid < 4) {
            float v = a[0];                    // (no dynamic index into registers)
#pragma unroll
            for (int c = 1; c < 4; ++c) v = tid == c ? a[c] : v;
            mine[tid] = v;
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(done, 1) == segs - 1;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        const float *all = sums + (int64_t)first * (4 + F);
#pragma unroll
        for (int c = 0; c < 4; ++c) a[c] = 0.f;
        for (int q = 0; q < segs; ++q)
#pragma unroll
            for (int c = 0; c < 4; ++c) a[c] += __ldcg(all + (int64_t)q * (4 + F) + c);
        for (int j = tid; j < F; j += FTH) {
            float x = 0.f;
#pragma unroll 4
            for (int q = 0; q < segs; ++q) x += __ldcg(all + (int64_t)q * (4 + F) + 4 + j);
            out_feat[(int64_t)g * F + j] = a[3] > 0.f ? x / a[3] : 0.f;
        }
    }
    const float W = a[3];
    const bool own = W > 0.f;
    const float mean[3] = {mg[0] + a[0] / W, mg[1] + a[1] / W, mg[2] + a[2] / W};
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    float cv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto add = [&](int s) {
        const float w = sl.w(s), d[3] = {sl.mu(s, 0) - mean[0], sl.mu(s, 1) - mean[1], sl.mu(s, 2) - mean[2]};
#pragma unroll
        for (int c = 0; c < 6; ++c) cv[c] += w * (sl.cv(s, c) + d[ia[c]] * d[ib[c]]);
    };
    if (tid == 0) add(g);
#pragma unroll 2
    for (int k = tid; k < m; k += FTH) add(mem[k]);
    block_sum<6>(cv, s_red, lane, warp);
    if (tid == 0) {
        out_w[g] = own ? W : 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) out_mu[(int64_t)c * T + g] = own ? mean[c] : 0.f;
#pragma unroll
        for (int c = 0; c < 6; ++c) out_cov[(int64_t)c * T + g] = own ? cv[c] / W : 0.f;
    }
}

// out_w, out_mu, out_cov and out_feat of every slot, a warp each: zeros for a
// merged one, the slot's own values for a winner without members, sums over the
// members (listed at members + off) otherwise.  The first BIG_BLOCKS blocks take
// the work items of the winners of more than BIG_MEMBERS members.  Bound by the
// gather of the members' rows: with one block per such winner and its members'
// loads one after the other, 100,000 detections of 70 entities (F = 64) took
// 1,734 us here and 300,000 of 40 11.4 ms; in segments with several loads in
// flight per lane 51 and 159.  (64 registers: a kernel of its own for them, with more
// loads in flight, costs every call a launch that mostly finds nothing, 3 us.)
__global__ void __launch_bounds__(FTH, 4)
assoc_fuse_kernel(Slots sl, const int32_t *__restrict__ parent, const int32_t *__restrict__ mcnt,
                  const int32_t *__restrict__ off, const int32_t *__restrict__ members, const int2 *__restrict__ items,
                  const int32_t *__restrict__ n_items, int32_t *done, float *sums, float *__restrict__ out_w,
                  float *__restrict__ out_mu, float *__restrict__ out_cov, float *__restrict__ out_feat, int vec)
{
    if (blockIdx.x < BIG_BLOCKS) {
        const int count = *n_items;
        for (int k = blockIdx.x; k < count; k += BIG_BLOCKS) {
            const int2 it = items[k];
            fuse_big(sl, it.x, it.y, k, members + off[it.x], mcnt[it.x], done + it.x, sums, vec, out_w, out_mu,
                     out_cov, out_feat);
            __syncthreads();             // the next segment reuses the shared arrays
        }
        return;
    }
    const int T = sl.N + sl.B, F = sl.F;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    const int t = (blockIdx.x - BIG_BLOCKS) * FW + warp;
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
}

}  // namespace

cudaError_t launch_assoc_init(const AssocArgs &a, cudaStream_t s)
{
    const int32_t T = a.N + a.B;
    assoc_init_kernel<<<(unsigned)((T + 255) / 256), 256, 0, s>>>(T, a.N, a.B, a.tau_f, a.label, a.win, a.mcnt, a.counters,
                                                                   a.emit.tau_key, a.emit.cnt, a.emit.cap, a.dhi,
                                                                   a.ehi, a.F_pad, a.probe);
    return cudaGetLastError();
}

cudaError_t launch_assoc_match(const AssocArgs &a, cudaStream_t s)
{
    assoc_match_kernel<<<(unsigned)a.B, TA, 0, s>>>(a.emit, a.N, a.B, a.ent_mu, a.ent_cov, a.ent_active, a.det_mu,
                                                    a.det_cov, a.h_max, a.max_m, a.match_cnt, a.match_idx, a.match_h,
                                                    a.label, a.counters + 1, a.over,
                                                    OverRows{a.dhi, a.dlo, a.chi, a.clo, a.F_pad}, a.err);
    return cudaGetLastError();
}

cudaError_t launch_assoc(const AssocArgs &a, cudaStream_t s)
{
    const int32_t N = a.N, B = a.B, T = a.N + a.B;
    if (B < 1 || N < 0 || a.F < 1 || a.max_m < 1 || (int64_t)B * a.max_m > 0x7fffffff) return cudaErrorInvalidValue;
    cudaError_t e;
    // the stored rows: all of them, or those the emitted lists overflowed for
    const int32_t *over = a.emit.cnt ? a.over : nullptr;
    const unsigned grid = (unsigned)(over && B > 1368 ? 1368 : B);     // (nine CTAs to an SM)
    assoc_search_kernel<<<grid, TA, 0, s>>>(a.S, a.ld, N, B, a.ent_mu, a.ent_cov, a.ent_active, a.det_mu, a.det_cov,
                                            a.tau_f, a.h_max, a.max_m, a.match_cnt, a.match_idx, a.match_h, a.label,
                                            a.counters + 1, over, a.counters + kAssocTicket, a.err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned nb = (unsigned)((T + 255) / 256);
    assoc_winner_kernel<<<nb, 256, 0, s>>>(N, T, a.ent_w, a.label, a.members, a.win);    // (roots: before the members)
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_parent_kernel<<<nb, 256, 0, s>>>(T, a.members, a.win, a.parent, a.mcnt, a.pos);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_offset_kernel<<<nb, 256, 0, s>>>(T, a.mcnt, a.off, a.pos, a.counters, a.items);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    assoc_members_kernel<<<nb, 256, 0, s>>>(T, a.parent, a.off, a.pos, a.members);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const Slots sl{N, B, a.F, a.ent_mu, a.ent_cov, a.ent_feat, a.ent_w, a.det_mu, a.det_cov, a.det_feat};
    const uintptr_t al = (uintptr_t)a.ent_feat | (uintptr_t)a.det_feat | (uintptr_t)a.out_feat;
    const int vec = a.F % 4 == 0 && (al & 15u) == 0 ? 1 : 0;
    assoc_fuse_kernel<<<(unsigned)((T + FW - 1) / FW + BIG_BLOCKS), FTH, 0, s>>>(
        sl, a.parent, a.mcnt, a.off, a.members, a.items, a.counters + kAssocItems, a.pos, a.sums, a.out_w, a.out_mu,
        a.out_cov, a.out_feat, vec);
    return cudaGetLastError();
}

}  // namespace farm
