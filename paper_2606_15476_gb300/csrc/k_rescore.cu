// k_rescore.cu -- FP32 re-scoring of the reduced-precision path's candidates.
//
// The BF16 similarity stage ranks every object approximately; for each row
// its C best objects are then re-scored with exact FP32 dot products of the
// unit rows (App. D.2 step 3 cosines) and the R best of them, in rank order
// (cosine descending, lower index first), become the row's rank list.  The
// result equals the FP32 path's list whenever the FP32 top R lie within the
// BF16 top C.
//
// Only the borderline candidates are re-scored: with the reduced-precision
// values of the (descending) candidate list at hand, a candidate whose value
// lies more than `band` below the R-th value is skipped (it would need an
// arithmetic error above the band to belong to the top R).
//
// Rows of a scene that ran the FP32-accurate similarity in the same batch
// (Piece::exact) already hold their final lists: copy_lists_kernel copies
// them, a warp per row.
//
// The work is a gather of whole descriptor rows (4.6 KB at D = 1152): the rows
// of one class of objects list mostly the same candidates, so a block takes
// four rows that are neighbours in an order by class and loads each candidate
// of their union once (rescore_group_kernel; launches of few rows take a row
// per block).  At 100,000 objects, D = 1152: 1.35 ms against 1.98 with a row
// per block (lists of 512 / 128, 6,001 target and 15,105 landmark rows, then
// bound by DRAM at 74% of its peak), 1.41 against 2.20 (lists of 256 / 64,
// 16,384 and 40,900 rows).  Rows longer than kGroupDimMax floats: a row per block, two
// candidates per warp step.
#include "farm_internal.h"

namespace farm {
namespace {

constexpr int TH = 256;
constexpr int SORT_MAX = 1024;

__device__ __forceinline__ uint32_t order_key(float f)
{
    const uint32_t u = __float_as_uint(f + 0.0f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_value(uint32_t k)
{
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

constexpr int kWarps = TH / 32;
constexpr int kGroupDimMax = 2048;          // longest rows (floats) the grouped kernel stages
// Rows a block takes together, and the launch size from which it does: below
// it a row per block keeps more SMs busy (2,048 rows are 512 blocks of four).
constexpr int kGroupRows = 4;
constexpr int64_t kGroupFrom = 2048;
constexpr int kBuckets = 4096;              // of the processing order's counting sort

// Dynamic shared memory of a block of G rows with lists of at most cmax:
// the unit rows; the union's hash table (object, a byte of row bits), whose
// place the rows' keys take once the union is listed; the union's list.
struct GroupSmem {
    size_t q, hkey, hmask, key, obj, mask, bytes;
    int H;
    __host__ __device__ GroupSmem(int dim_pad, int G, int cmax)
    {
        auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
        const int E = G * cmax;
        H = 64;
        while (G > 1 && H < E + (E >> 1)) H <<= 1;
        q = 0;
        hkey = up(q + (size_t)G * dim_pad * 4);
        hmask = hkey + (size_t)H * 4;
        key = hkey;
        const size_t a = up(hmask + H), k = up(key + (size_t)E * 8);
        obj = a > k ? a : k;
        mask = up(obj + (size_t)E * 4);
        bytes = up(mask + E);
    }
};

// What a block needs of one of its rows.
struct GroupRow {
    const float *d32;
    int64_t co;              // its list's offset
    int64_t oo;              // its output list's offset
    int64_t q_row;
    float thr;               // candidates valued below it are out of the band
    int32_t C, R, n_obj, tgt;
};

__device__ __forceinline__ int find_row_piece(const Piece *__restrict__ pieces, int n_pieces, int64_t r)
{
    int lo = 0, hi = n_pieces - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pieces[mid].row_begin <= r) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The R best of the n distinct keys of one row (shared memory, n <= 32 REG),
// by one warp, into oi / oc in rank order, -1 / 0 past them.  The R-th largest
// 32-bit value key T by a bitwise search below the leading bits that the
// smallest and largest share (stopped once exactly R keys reach the
// candidate); the words reaching T gathered in place; those ranked by counting.
template <int REG>
__device__ __forceinline__ void warp_rank_out(uint64_t *key, int n, int R, int32_t *__restrict__ oi,
                                              float *__restrict__ oc, int out_stride, int lane)
{
    const unsigned FULL = 0xffffffffu;
    uint64_t w[REG];
    uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
    for (int k = 0; k < REG; ++k) {
        const int t = lane + 32 * k;
        w[k] = t < n ? key[t] : 0ull;          // (no real word is 0: its key would encode a NaN)
        if (t < n) {
            kmin = min(kmin, (uint32_t)(w[k] >> 32));
            kmax = max(kmax, (uint32_t)(w[k] >> 32));
        }
    }
    kmin = __reduce_min_sync(FULL, kmin);
    kmax = __reduce_max_sync(FULL, kmax);
    const int keep = min(n, min(R, out_stride));
    uint32_t T = 0u;
    if (n > keep) {
        const uint32_t diff = kmin ^ kmax;
        const int top = diff ? 31 - __clz(diff) : -1;
        T = top < 0 ? kmin : (top == 31 ? 0u : kmin & ~((2u << top) - 1u));
#pragma unroll 1
        for (int bit = top; bit >= 0; --bit) {
            const uint32_t c = T | (1u << bit);
            int cnt = 0;
#pragma unroll
            for (int k = 0; k < REG; ++k) cnt += (uint32_t)(w[k] >> 32) >= c ? 1 : 0;
            cnt = (int)__reduce_add_sync(FULL, (unsigned)cnt);
            if (cnt >= keep) {
                T = c;
                if (cnt == keep) break;        // no lower bit changes which words reach T
            }
        }
    }
    __syncwarp();                              // every lane holds its words before they are overwritten
    int nc = 0;
#pragma unroll
    for (int k = 0; k < REG; ++k) {
        const bool take = w[k] != 0ull && (uint32_t)(w[k] >> 32) >= T;
        const unsigned bal = __ballot_sync(FULL, take);
        if (take) key[nc + __popc(bal & ((1u << lane) - 1u))] = w[k];
        nc += __popc(bal);
    }
    __syncwarp();
    for (int j = lane; j < nc; j += 32) {
        const uint64_t x = key[j];
        int c = 0;
        for (int t = 0; t < nc; ++t) c += key[t] > x ? 1 : 0;
        if (c < keep) {
            oi[c] = (int32_t)(0xffffffffu - (uint32_t)(x & 0xffffffffu));
            if (oc) oc[c] = key_value((uint32_t)(x >> 32));
        }
    }
    for (int k = keep + lane; k < out_stride; k += 32) {
        oi[k] = -1;
        if (oc) oc[k] = 0.f;
    }
}

// One step of the warp's sums of NV values at once: each half of the lanes
// keeps half of the values (the sums pair the same lanes as a butterfly per
// value would, so they are bitwise those).
template <int NV>
__device__ __forceinline__ void fold_sums(float *v, int lane, int o)
{
    if constexpr (NV == 1) {
        for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    } else {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < NV / 2; ++k) {
            const float keep = up ? v[k + NV / 2] : v[k];
            const float send = up ? v[k] : v[k + NV / 2];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        fold_sums<NV / 2>(v, lane, o >> 1);
    }
}

// G rows of the processing order per block (rows of up to kGroupDimMax
// floats).  Rows of one class of objects list mostly the same candidates, and
// what bounds the work is the bytes of their descriptor rows: the block takes
// the union of its rows' in-band candidates, loads each one once (two per
// warp in flight, straight into registers) and multiplies it with every row
// that lists it.  Each dot product has the order of a row on its own: lane l
// adds the products of float4 l, l + 32, ..., then the lanes' sums are added
// in a butterfly.
template <int G>
__global__ void __launch_bounds__(TH, 4)
rescore_group_kernel(const Piece *__restrict__ pieces, int32_t n_pieces, int64_t total_rows,
                     const int32_t *__restrict__ order, const float *__restrict__ Q32, int32_t dim_pad,
                     const int32_t *__restrict__ bsel_t, const float *__restrict__ bsel_tv, int32_t cstride_t,
                     const int32_t *__restrict__ bsel_l, const float *__restrict__ bsel_lv, int32_t cstride_l,
                     float band, int32_t *__restrict__ tsel_idx, float *__restrict__ tsel_cos, int32_t stride_t,
                     int32_t *__restrict__ lsel_idx, int32_t stride_l, int cmax)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const GroupSmem L(dim_pad, G, cmax);
    float4 *q4 = reinterpret_cast<float4 *>(sm + L.q);
    int32_t *hkey = reinterpret_cast<int32_t *>(sm + L.hkey);
    uint32_t *hmask = reinterpret_cast<uint32_t *>(sm + L.hmask);     // four byte masks per word
    uint64_t *key = reinterpret_cast<uint64_t *>(sm + L.key);         // [G][cmax], after the union is listed
    int32_t *uobj = reinterpret_cast<int32_t *>(sm + L.obj);
    uint8_t *umask = sm + L.mask;
    __shared__ GroupRow rows[G];
    __shared__ int s_n, s_cnt[G];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nv = dim_pad >> 2;
    const int64_t p0 = (int64_t)blockIdx.x * G;
    if (tid < G) {
        GroupRow w{};
        if (p0 + tid < total_rows) {
            const int64_t r = order ? order[p0 + tid] : p0 + tid;
            const Piece &pc = pieces[find_row_piece(pieces, n_pieces, r)];
            const int i = (int)(r - pc.row_begin);
            const bool tgt = i < pc.ntr;
            const int64_t l = pc.l_row0 + (i - pc.ntr);
            w.d32 = pc.d32;
            w.co = tgt ? (pc.t_row0 + i) * (int64_t)cstride_t : l * (int64_t)cstride_l;
            w.oo = tgt ? (pc.t_row0 + i) * (int64_t)stride_t : l * (int64_t)stride_l;
            w.q_row = pc.q_row0 + i;
            w.C = tgt ? pc.fkeep_t : pc.fkeep_l;
            w.R = tgt ? pc.R : pc.klm;
            w.n_obj = pc.n_obj;
            w.tgt = tgt;
            const float *vals = tgt ? bsel_tv : bsel_lv;
            w.thr = vals ? vals[w.co + w.R - 1] - band : -__int_as_float(0x7f800000);
        }
        rows[tid] = w;
    }
    __syncthreads();
    for (int g = 0; g < G; ++g) {
        if (!rows[g].d32) continue;
        const float4 *src = reinterpret_cast<const float4 *>(Q32 + rows[g].q_row * (int64_t)dim_pad);
        for (int i = tid; i < nv; i += TH) q4[g * nv + i] = src[i];
    }
    // the rows of one scene at a time (as a rule all of them)
    uint32_t todo = 0u;
    for (int g = 0; g < G; ++g) todo |= rows[g].d32 ? 1u << g : 0u;
    while (todo) {
        const float *D32 = rows[__ffs(todo) - 1].d32;
        uint32_t sub = 0u;
        for (int g = 0; g < G; ++g) sub |= ((todo >> g) & 1u) && rows[g].d32 == D32 ? 1u << g : 0u;
        todo &= ~sub;
        if (G > 1) {
            for (int s = tid; s < L.H; s += TH) hkey[s] = -1;
            for (int s = tid; s < L.H / 4; s += TH) hmask[s] = 0u;
        }
        if (tid == 0) s_n = 0;
        if (tid < G) s_cnt[tid] = 0;
        __syncthreads();
        // the union of the rows' in-band candidates (an index outside the scene is dropped)
        for (int g = 0; g < G; ++g) {
            if (!((sub >> g) & 1u)) continue;
            const int32_t *cr = (rows[g].tgt ? bsel_t : bsel_l) + rows[g].co;
            const float *vals = rows[g].tgt ? bsel_tv : bsel_lv;
            const float *cv = vals ? vals + rows[g].co : nullptr;
            const float thr = rows[g].thr;
            const int C = rows[g].C, n_obj = rows[g].n_obj;
            for (int c0 = warp * 32; c0 < C; c0 += TH) {
                const int c = c0 + lane;
                const int32_t e = c < C ? cr[c] : -1;
                const bool in = c < C && !(cv && cv[c] < thr) && e >= 0 && e < n_obj;
                if (G == 1) {
                    const uint32_t m = __ballot_sync(0xffffffffu, in);
                    int base = 0;
                    if (lane == 0 && m) base = atomicAdd(&s_n, __popc(m));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (in) {
                        const int at = base + __popc(m & ((1u << lane) - 1u));
                        uobj[at] = e;
                        umask[at] = 1;
                    }
                } else if (in) {
                    // (at most G cmax distinct objects in a table of at least half as many more slots)
                    uint32_t s = ((uint32_t)e * 2654435761u) & (uint32_t)(L.H - 1);
                    for (int t = 0; t < L.H; ++t) {
                        const int32_t old = atomicCAS(&hkey[s], -1, e);
                        if (old == -1 || old == e) {
                            atomicOr(&hmask[s >> 2], 1u << (8 * (s & 3u) + g));
                            break;
                        }
                        s = (s + 1) & (uint32_t)(L.H - 1);
                    }
                }
            }
        }
        __syncthreads();
        if (G > 1) {
            for (int s = tid; s < L.H; s += TH) {       // (H is a multiple of the warp)
                const int32_t e = hkey[s];
                const uint32_t m = __ballot_sync(0xffffffffu, e >= 0);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&s_n, __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (e >= 0) {
                    const int at = base + __popc(m & ((1u << lane) - 1u));
                    uobj[at] = e;
                    umask[at] = (uint8_t)(hmask[s >> 2] >> (8 * (s & 3)));
                }
            }
            __syncthreads();
        }
        const int n = s_n;
        constexpr int U = 3;                // float4 of each candidate in flight per lane
        for (int p = 2 * warp; p < n; p += 2 * kWarps) {
            const bool two = p + 1 < n;
            const int32_t e0 = uobj[p], e1 = uobj[two ? p + 1 : p];
            const uint32_t m0 = umask[p], m1 = two ? umask[p + 1] : 0u, mm = m0 | m1;
            const float4 *x0 = reinterpret_cast<const float4 *>(D32 + (int64_t)e0 * dim_pad);
            const float4 *x1 = reinterpret_cast<const float4 *>(D32 + (int64_t)e1 * dim_pad);
            float acc[2 * G];
#pragma unroll
            for (int k = 0; k < 2 * G; ++k) acc[k] = 0.f;
            for (int base = 0; base < nv; base += 32 * U) {
                float4 a[U], b[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = base + u * 32 + lane;
                    a[u] = i < nv ? __ldg(x0 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                    b[u] = i < nv ? __ldg(x1 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = base + u * 32 + lane;
                    if (i >= nv) continue;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (G > 1 && !((mm >> g) & 1u)) continue;       // (warp-uniform)
                        const float4 y = q4[g * nv + i];
                        acc[g] = fmaf(y.x, a[u].x, acc[g]);
                        acc[g] = fmaf(y.y, a[u].y, acc[g]);
                        acc[g] = fmaf(y.z, a[u].z, acc[g]);
                        acc[g] = fmaf(y.w, a[u].w, acc[g]);
                        acc[G + g] = fmaf(y.x, b[u].x, acc[G + g]);
                        acc[G + g] = fmaf(y.y, b[u].y, acc[G + g]);
                        acc[G + g] = fmaf(y.z, b[u].z, acc[G + g]);
                        acc[G + g] = fmaf(y.w, b[u].w, acc[G + g]);
                    }
                }
            }
            fold_sums<2 * G>(acc, lane, 16);
            // the lane's value is that of candidate (lane bit 4) and row (the bits
            // below it), held by 32 / 2G lanes
            constexpr int REP = 32 / (2 * G);
            const int which = lane / REP;
            const int c = which / G, g = which % G;
            if ((lane % REP) == 0 && (((c ? m1 : m0) >> g) & 1u)) {
                const int32_t e = c ? e1 : e0;
                key[g * cmax + atomicAdd(&s_cnt[g], 1)] =
                    ((uint64_t)order_key(acc[0]) << 32) | (uint64_t)(0xffffffffu - (uint32_t)e);
            }
        }
        __syncthreads();
        // the rows' lists, a warp per row
        for (int g = warp; g < G; g += kWarps) {
            if (!((sub >> g) & 1u)) continue;
            const bool tgt = rows[g].tgt != 0;
            int32_t *oi = (tgt ? tsel_idx : lsel_idx) + rows[g].oo;
            float *oc = tgt && tsel_cos ? tsel_cos + rows[g].oo : nullptr;
            const int stride = tgt ? stride_t : stride_l;
            const int m = s_cnt[g], R = rows[g].R;
            uint64_t *kg = key + g * cmax;
            if (m <= 128) warp_rank_out<4>(kg, m, R, oi, oc, stride, lane);
            else if (m <= 256) warp_rank_out<8>(kg, m, R, oi, oc, stride, lane);
            else warp_rank_out<kMaxTargetCands / 32>(kg, m, R, oi, oc, stride, lane);
        }
        if (todo) __syncthreads();       // the next scene's rows reuse the table
    }
}

// The processing order of a grouped launch: its rows by the class of their
// best candidate (a counting sort by a hash of class and piece; the order
// within a bucket is free, and so is the whole order as far as results go), so
// that a block's rows and its neighbours' list mostly the same objects.
__global__ void __launch_bounds__(256)
rescore_bucket_kernel(const Piece *__restrict__ pieces, int32_t n_pieces, int32_t rows,
                      const int32_t *__restrict__ bsel_t, int32_t cstride_t, const int32_t *__restrict__ bsel_l,
                      int32_t cstride_l, int32_t *__restrict__ hist, int2 *__restrict__ place)
{
    const int r = blockIdx.x * 256 + threadIdx.x;
    if (r >= rows) return;
    const int k = find_row_piece(pieces, n_pieces, r);
    const Piece &pc = pieces[k];
    const int i = (int)(r - pc.row_begin);
    const int32_t e = i < pc.ntr ? bsel_t[(pc.t_row0 + i) * (int64_t)cstride_t]
                                 : bsel_l[(pc.l_row0 + (i - pc.ntr)) * (int64_t)cstride_l];
    const int32_t c = e >= 0 && e < pc.n_obj ? pc.cls[e] : -1;
    const int b = (int)(((uint32_t)c + (uint32_t)k * 7919u) & (uint32_t)(kBuckets - 1));
    place[r] = make_int2(b, atomicAdd(&hist[b], 1));
}

__global__ void __launch_bounds__(256)
rescore_order_kernel(int32_t rows, const int32_t *__restrict__ hist, const int2 *__restrict__ place,
                     int32_t *__restrict__ order)
{
    __shared__ int32_t base[kBuckets];
    __shared__ int32_t wsum[8];
    constexpr int PER = kBuckets / 256;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t v[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = hist[tid * PER + k];
        sum += v[k];
    }
    int32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int32_t at = incl - sum;
    for (int w = 0; w < warp; ++w) at += wsum[w];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        base[tid * PER + k] = at;
        at += v[k];
    }
    __syncthreads();
    const int r = blockIdx.x * 256 + tid;
    if (r < rows) {
        const int2 p = place[r];
        order[base[p.x] + p.y] = r;
    }
}

// One row, loads from global memory: the C candidates cr (values cv, nullable) against the unit row q
// (global, dim_pad floats) -> the R best in rank order into oi / oc.
__device__ __forceinline__ void rescore_row_ldg(const float *__restrict__ q, int32_t dim_pad,
                                            const float *__restrict__ D32, const int32_t *__restrict__ cr,
                                            const float *__restrict__ cv, float band, int32_t C, int32_t R,
                                            int32_t *__restrict__ oi, float *__restrict__ oc, int32_t out_stride)
{
    extern __shared__ float4 q4[];
    __shared__ uint64_t key[SORT_MAX];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nv = dim_pad / 4;
    const float4 *src = reinterpret_cast<const float4 *>(q);
    for (int i = tid; i < nv; i += TH) q4[i] = src[i];
    __syncthreads();
    const float thr = cv ? cv[R - 1] - band : 0.f;
    // two candidates per warp step, four float4 loads of each in flight per lane
    for (int c0 = 2 * warp; c0 < C; c0 += 2 * (TH / 32)) {
        const int c1 = c0 + 1;
        const bool do0 = !(cv && cv[c0] < thr);
        const bool do1 = c1 < C && !(cv && cv[c1] < thr);
        if (!do0 && !do1) {
            if (lane == 0) {
                key[c0] = 0ull;
                if (c1 < C) key[c1] = 0ull;
            }
            continue;
        }
        const int32_t e0 = do0 ? cr[c0] : 0, e1 = do1 ? cr[c1] : 0;
        const float4 *p0 = reinterpret_cast<const float4 *>(D32 + (int64_t)e0 * dim_pad);
        const float4 *p1 = reinterpret_cast<const float4 *>(D32 + (int64_t)e1 * dim_pad);
        float a0 = 0.f, a1 = 0.f;
        for (int base = 0; base < nv; base += 4 * 32) {
            float4 x0[4], x1[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + u * 32 + lane;
                const bool in = i < nv;
                x0[u] = (in && do0) ? __ldg(p0 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                x1[u] = (in && do1) ? __ldg(p1 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + u * 32 + lane;
                if (i < nv) {
                    const float4 q = q4[i];
                    a0 = fmaf(q.x, x0[u].x, a0);
                    a0 = fmaf(q.y, x0[u].y, a0);
                    a0 = fmaf(q.z, x0[u].z, a0);
                    a0 = fmaf(q.w, x0[u].w, a0);
                    a1 = fmaf(q.x, x1[u].x, a1);
                    a1 = fmaf(q.y, x1[u].y, a1);
                    a1 = fmaf(q.z, x1[u].z, a1);
                    a1 = fmaf(q.w, x1[u].w, a1);
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
        }
        if (lane == 0) {
            key[c0] = do0 ? ((uint64_t)order_key(a0) << 32) | (uint64_t)(0xffffffffu - (uint32_t)e0) : 0ull;
            if (c1 < C) key[c1] = do1 ? ((uint64_t)order_key(a1) << 32) | (uint64_t)(0xffffffffu - (uint32_t)e1) : 0ull;
        }
    }
    int P = 1;
    while (P < C) P <<= 1;
    for (int i = C + tid; i < P; i += TH) key[i] = 0ull;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < P; i += TH) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const uint64_t a = key[i], b = key[ixj];
                    const bool desc = (i & k) == 0;
                    if (desc ? (a < b) : (a > b)) { key[i] = b; key[ixj] = a; }
                }
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < out_stride; i += TH) {
        if (i < R) {
            oi[i] = (int32_t)(0xffffffffu - (uint32_t)(key[i] & 0xffffffffu));
            if (oc) oc[i] = key_value((uint32_t)(key[i] >> 32));
        } else {
            oi[i] = -1;
            if (oc) oc[i] = 0.f;
        }
    }
}

// Rows longer than kGroupDimMax: a row per block, found through the piece table.
__global__ void __launch_bounds__(TH)
rescore_grouped_kernel(const Piece *__restrict__ pieces, int32_t n_pieces, const float *__restrict__ Q32,
                       int32_t dim_pad, const int32_t *__restrict__ bsel_t, const float *__restrict__ bsel_tv,
                       int32_t cstride_t, const int32_t *__restrict__ bsel_l, const float *__restrict__ bsel_lv,
                       int32_t cstride_l, float band, int32_t *__restrict__ tsel_idx, float *__restrict__ tsel_cos,
                       int32_t stride_t, int32_t *__restrict__ lsel_idx, int32_t stride_l)
{
    const int64_t r = blockIdx.x;
    const Piece pc = pieces[find_piece(pieces, n_pieces, r, [](const Piece &x) { return x.row_begin; })];
    const int i = (int)(r - pc.row_begin);
    const float *q = Q32 + (pc.q_row0 + i) * (int64_t)dim_pad;
    const bool tgt = i < pc.ntr;
    const int64_t l = pc.l_row0 + (i - pc.ntr);
    const int64_t co = tgt ? (pc.t_row0 + i) * (int64_t)cstride_t : l * (int64_t)cstride_l;
    const int32_t *cr = (tgt ? bsel_t : bsel_l) + co;
    const float *vals = tgt ? bsel_tv : bsel_lv;
    const float *cv = vals ? vals + co : nullptr;
    const int32_t C = tgt ? pc.fkeep_t : pc.fkeep_l, R = tgt ? pc.R : pc.klm;
    int32_t *oi = tgt ? tsel_idx + (pc.t_row0 + i) * (int64_t)stride_t : lsel_idx + l * (int64_t)stride_l;
    float *oc = tgt && tsel_cos ? tsel_cos + (pc.t_row0 + i) * (int64_t)stride_t : nullptr;
    const int32_t out = tgt ? stride_t : stride_l;
    rescore_row_ldg(q, dim_pad, pc.d32, cr, cv, band, C, R, oi, oc, out);
}

// The final lists of launch rows [row0, row0 + rows) -- rows of FP32-accurate
// scenes -- copied from the candidate buffers: R (klm) entries, -1 / 0 past them.
__global__ void __launch_bounds__(256)
copy_lists_kernel(const Piece *__restrict__ pieces, int32_t n_pieces, int64_t row0, int64_t rows,
                  const int32_t *__restrict__ bsel_t, const float *__restrict__ bsel_tv, int32_t cstride_t,
                  const int32_t *__restrict__ bsel_l, int32_t cstride_l, int32_t *__restrict__ tsel_idx,
                  float *__restrict__ tsel_cos, int32_t stride_t, int32_t *__restrict__ lsel_idx, int32_t stride_l)
{
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (w >= rows) return;
    const int64_t r = row0 + w;
    int lo = 0;
    if (lane == 0) {
        int hi = n_pieces - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pieces[mid].row_begin <= r) lo = mid;
            else hi = mid - 1;
        }
    }
    const Piece &pc = pieces[__shfl_sync(0xffffffffu, lo, 0)];
    const int i = (int)(r - pc.row_begin);
    const bool tgt = i < pc.ntr;
    const int64_t l = pc.l_row0 + (i - pc.ntr);
    const int64_t co = tgt ? (pc.t_row0 + i) * (int64_t)cstride_t : l * (int64_t)cstride_l;
    const int32_t *src = (tgt ? bsel_t : bsel_l) + co;
    int32_t *oi = tgt ? tsel_idx + (pc.t_row0 + i) * (int64_t)stride_t : lsel_idx + l * (int64_t)stride_l;
    float *oc = tgt && tsel_cos ? tsel_cos + (pc.t_row0 + i) * (int64_t)stride_t : nullptr;
    const int keep = tgt ? pc.R : pc.klm, out = tgt ? stride_t : stride_l;
    for (int k = lane; k < out; k += 32) {
        oi[k] = k < keep ? src[k] : -1;
        if (oc) oc[k] = k < keep ? bsel_tv[co + k] : 0.f;
    }
}

}  // namespace

cudaError_t launch_copy_lists(const Piece *pieces, int32_t n_pieces, int64_t row0, int64_t rows, const int32_t *bsel_t,
                              const float *bsel_tv, int32_t cstride_t, const int32_t *bsel_l, int32_t cstride_l,
                              int32_t *tsel_idx, float *tsel_cos, int32_t stride_t, int32_t *lsel_idx,
                              int32_t stride_l, cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    if (n_pieces < 1 || (tsel_cos && !bsel_tv)) return cudaErrorInvalidValue;
    const int64_t blocks = (rows + 7) / 8;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    copy_lists_kernel<<<(unsigned)blocks, 256, 0, s>>>(pieces, n_pieces, row0, rows, bsel_t, bsel_tv, cstride_t,
                                                        bsel_l, cstride_l, tsel_idx, tsel_cos, stride_t, lsel_idx,
                                                        stride_l);
    return cudaGetLastError();
}

size_t rescore_scratch_ints(int64_t rows)
{
    return rows >= kGroupFrom ? (size_t)kBuckets + 3 * (size_t)rows : 0;
}

cudaError_t launch_rescore_grouped(const Piece *pieces, int32_t n_pieces, int64_t total_rows, const float *Q32,
                                   int32_t dim_pad, const int32_t *bsel_t, const float *bsel_tv, int32_t cstride_t,
                                   const int32_t *bsel_l, const float *bsel_lv, int32_t cstride_l, float band,
                                   int32_t *tsel_idx, float *tsel_cos, int32_t stride_t, int32_t *lsel_idx,
                                   int32_t stride_l, int32_t *scratch, cudaStream_t s)
{
    if (total_rows <= 0) return cudaSuccess;
    if (n_pieces < 1 || total_rows > 0x7fffffff || dim_pad % 4 != 0 || cstride_t > kMaxTargetCands ||
        cstride_l > kMaxTargetCands)
        return cudaErrorInvalidValue;
    const int cmax = cstride_t > cstride_l ? cstride_t : cstride_l;
    const bool group = total_rows >= kGroupFrom;
    cudaError_t e;
    if (dim_pad > kGroupDimMax) {
        const size_t smem = (size_t)dim_pad * sizeof(float);
        if (smem > 48 * 1024 &&
            (e = cudaFuncSetAttribute(rescore_grouped_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem)) != cudaSuccess)
            return e;
        rescore_grouped_kernel<<<(unsigned)total_rows, TH, smem, s>>>(pieces, n_pieces, Q32, dim_pad, bsel_t, bsel_tv,
                                                                      cstride_t, bsel_l, bsel_lv, cstride_l, band,
                                                                      tsel_idx, tsel_cos, stride_t, lsel_idx, stride_l);
        return cudaGetLastError();
    }
    int32_t *order = nullptr;
    if (group) {
        if (!scratch) return cudaErrorInvalidValue;
        int32_t *hist = scratch;
        int2 *place = reinterpret_cast<int2 *>(scratch + kBuckets);
        order = scratch + kBuckets + 2 * total_rows;
        if ((e = cudaMemsetAsync(hist, 0, kBuckets * sizeof(int32_t), s)) != cudaSuccess) return e;
        const unsigned nb = (unsigned)((total_rows + 255) / 256);
        rescore_bucket_kernel<<<nb, 256, 0, s>>>(pieces, n_pieces, (int32_t)total_rows, bsel_t, cstride_t, bsel_l,
                                                 cstride_l, hist, place);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        rescore_order_kernel<<<nb, 256, 0, s>>>((int32_t)total_rows, hist, place, order);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int G = group ? kGroupRows : 1;
    const size_t smem = GroupSmem(dim_pad, G, cmax).bytes;
    auto kern = group ? rescore_group_kernel<kGroupRows> : rescore_group_kernel<1>;
    if (smem + 1024 > 48 * 1024 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
                                cudaSuccess)
        return e;
    kern<<<(unsigned)((total_rows + G - 1) / G), TH, smem, s>>>(pieces, n_pieces, total_rows, order, Q32, dim_pad,
                                                                bsel_t, bsel_tv, cstride_t, bsel_l, bsel_lv, cstride_l,
                                                                band, tsel_idx, tsel_cos, stride_t, lsel_idx, stride_l,
                                                                cmax);
    return cudaGetLastError();
}

}  // namespace farm
