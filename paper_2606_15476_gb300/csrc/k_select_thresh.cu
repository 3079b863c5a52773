// k_select_thresh.cu -- thresholded rank selection over the similarity rows
// of the tensor-core paths (App. D.2 step 3 ranks, step 4 landmark
// candidates): the R largest entries of a row, in rank order.
//
// The similarity kernel's epilogue leaves, per row, the maximum of every
// group of 32 (8 in small scenes) consecutive objects.  Those values are
// entries of the row, so the R-th largest of their union, tau, is at most the
// row's R-th largest value: every entry of rank <= R has a value >= tau, and
// it lies in a group whose maximum is >= tau.  Only those groups (about R of
// them) are read: their entries >= tau are the candidates (the top R, their
// ties, and the few entries between tau and the R-th value when two of the
// top R share a group), and a sort of the candidates by (value desc, index
// asc) gives the exact rank list.  A row whose qualifying groups exceed the
// group list is streamed whole instead; a row whose candidates overflow the
// buffer is selected exactly by the global-memory radix select.
//
// Short rows (at most 2,048 objects) with fewer groups than R are staged whole
// in shared memory; their R-th largest key is found there and the candidates
// are taken from the staged keys.
//
// One CTA of 256 threads per row: the group maxima (at most 8,192 values) are
// staged in shared memory and the bound tau found by counting them into value
// bins; the candidates are ranked by value bins too (rank_words), so a row is a
// dozen barriers and no sort.  What bounds it is that chain and the gather of
// the groups: 100,000 objects, lists of 256: 231 us for 10,737 rows (22 ns a
// row, 2.3 TB/s of maxima and groups; the warp-per-row select it replaced took
// 360), lists of 64: 138 us (196); 20,000 objects, 1,024 lists of 321 and 2,546
// of 65: 54 us (110); 8,496 objects, lists of 95 and 16: 120 us for 15,169 rows
// (126).  (2,048 bins: 263, 157, 56 and 148 us: clearing and summing them.)
#include "select_common.cuh"

namespace farm {
namespace {

using namespace sel;

constexpr int TT = 256;
constexpr int CAP = 2048;          // candidate words per row before the exact fallback
constexpr int UNION_MAX = 8192;    // union values staged (a prefix of a longer union is still a subset)
constexpr int GLIST = 1024;        // qualifying groups gathered before the row is streamed whole
constexpr int BINS = 512;          // value bins of the bound and of the ranks
constexpr int BIN_BITS = 9;
constexpr int UNROLL = 4;          // float4 loads in flight per thread
constexpr int COUNT_MAX = 96;      // candidates ranked by counting each against all
constexpr int RANK_MAX = 768;      // candidates ranked by value bins; more are sorted

__device__ __forceinline__ void push_cand(uint64_t *cand, int *s_cnt, float x, int32_t j)
{
    const int pos = atomicAdd(s_cnt, 1);
    if (pos < CAP) cand[pos] = cand_word(order_key(x), j);
}

// Entries [j0, n) of the row compared against tau (float4 loads from a
// 16-byte aligned j0, scalar loads for the last n % 4).
__device__ __forceinline__ void stream_tail(const float *__restrict__ row, int j0, int n, float tau, uint64_t *cand,
                                            int *s_cnt)
{
    const int tid = threadIdx.x;
    const int n4 = n >> 2, g4 = j0 >> 2;
    const float4 *row4 = reinterpret_cast<const float4 *>(row);
    for (int g0 = g4; g0 < n4; g0 += TT * UNROLL) {
        float4 v[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int g = g0 + u * TT + tid;
            v[u] = g < n4 ? __ldcs(row4 + g) : make_float4(-1e30f, -1e30f, -1e30f, -1e30f);
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int g = g0 + u * TT + tid;
            if (g >= n4) continue;
            const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (x[c] >= tau) push_cand(cand, s_cnt, x[c], 4 * g + c);
        }
    }
    for (int j = max(4 * n4, j0) + tid; j < n; j += TT) {
        const float x = __ldcs(row + j);
        if (x >= tau) push_cand(cand, s_cnt, x, j);
    }
}

// A lower bound of the R-th largest of n keys in shared memory (n >= R >= 1;
// the caller has just written them) that at most `slack` more than R keys
// reach, or the R-th largest itself.  The keys between the smallest and the
// largest are counted in up to 512 equal bins (the group maxima of a row
// share their leading bits, so digits of the key itself would crowd a few
// bins), the bin of the R-th largest found, and refined while too many keys
// reach its lower edge: one pass as a rule.  s_mm: 2 TT / 32 words; top: the
// largest key.
__device__ __forceinline__ uint32_t kth_lower(const uint32_t *keys, int n, int R, int slack, uint32_t *hist,
                                              uint32_t *wsum, uint32_t *s3, uint32_t *s_mm, uint32_t &top)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int j = tid; j < n; j += TT) {       // (the thread's own keys: no barrier yet)
        lo = min(lo, keys[j]);
        hi = max(hi, keys[j]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        s_mm[2 * warp] = lo;
        s_mm[2 * warp + 1] = hi;
    }
    for (int i = tid; i < BINS; i += TT) hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < TT / 32; ++w) {
        lo = min(lo, s_mm[2 * w]);
        hi = max(hi, s_mm[2 * w + 1]);
    }
    uint32_t base = lo, span = hi - lo, remaining = (uint32_t)R;
    top = hi;
#pragma unroll 1
    for (;;) {
        const int bits = span ? 32 - __clz(span) : 0, shift = bits > BIN_BITS ? bits - BIN_BITS : 0;
        for (int j = tid; j < n; j += TT) {
            const uint32_t d = keys[j] - base;
            if (keys[j] >= base && d <= span) atomicAdd(&hist[d >> shift], 1u);
        }
        __syncthreads();
        find_bucket<BINS, TT>(hist, remaining, wsum, &s3[0], &s3[1], &s3[2]);
        const uint32_t bin = s3[0], rem = s3[1], cnt = s3[2];
        base += bin << shift;
        // R - rem keys lie above the bin, cnt in it
        if (shift == 0 || cnt - rem <= (uint32_t)slack) break;
        span = min(span - (bin << shift), (1u << shift) - 1u);
        remaining = rem;
        for (int i = tid; i < BINS; i += TT) hist[i] = 0;
        __syncthreads();
    }
    return base;
}

// The R best of the cnt distinct candidate words (cnt <= RANK_MAX, their keys in
// [T, top]) written in rank order.  Few: each one's rank counted against the
// others.  More: counted into 512 equal value bins, laid out bin by bin from
// the top, and ranked within their bin, which holds one or two as a rule.
__device__ __forceinline__ void rank_words(const uint64_t *cand, int cnt, int R, uint32_t T, uint32_t top,
                                           uint32_t *hist, uint32_t *wsum, uint64_t *sorted, int32_t *__restrict__ oi,
                                           float *__restrict__ oc)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto put = [&](uint64_t w, int r) {
        if (r >= R) return;
        oi[r] = (int32_t)(0xffffffffu - (uint32_t)(w & 0xffffffffu));
        if (oc) oc[r] = key_value((uint32_t)(w >> 32));
    };
    if (cnt <= COUNT_MAX) {
        for (int c = tid; c < cnt; c += TT) {
            const uint64_t w = cand[c];
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) r += cand[j] > w ? 1 : 0;
            put(w, r);
        }
        return;
    }
    const uint32_t span = top - T;
    const int bits = span ? 32 - __clz(span) : 0, shift = bits > BIN_BITS ? bits - BIN_BITS : 0;
    for (int i = tid; i < BINS; i += TT) hist[i] = 0;
    __syncthreads();
    for (int c = tid; c < cnt; c += TT) atomicAdd(&hist[((uint32_t)(cand[c] >> 32) - T) >> shift], 1u);
    __syncthreads();
    // each bin's first place: the entries of the higher bins
    constexpr int BPT = BINS / TT;
    uint32_t loc[BPT], sum = 0;
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        loc[i] = hist[BINS - 1 - (tid * BPT + i)];
        sum += loc[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t at = incl - sum;
    for (int w = 0; w < warp; ++w) at += wsum[w];
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        hist[BINS - 1 - (tid * BPT + i)] = at;
        at += loc[i];
    }
    __syncthreads();
    for (int c = tid; c < cnt; c += TT) {
        const uint64_t w = cand[c];
        sorted[atomicAdd(&hist[((uint32_t)(w >> 32) - T) >> shift], 1u)] = w;
    }
    __syncthreads();
    // (a bin's places now end at its counter and start at the next higher bin's)
    for (int c = tid; c < cnt; c += TT) {
        const uint64_t w = sorted[c];
        const uint32_t b = ((uint32_t)(w >> 32) - T) >> shift;
        const uint32_t e0 = b == BINS - 1u ? 0u : hist[b + 1], e1 = hist[b];
        int r = (int)e0;
        for (uint32_t k = e0; k < e1; ++k) r += sorted[k] > w ? 1 : 0;
        put(w, r);
    }
}

// The largest key of the candidates that may be ranked by bins, at least `top`:
// of a row whose group maxima are staged as a prefix, an entry past it may lie
// above them all.  (Out of line: only rows of more than UNION_MAX groups take it.)
__device__ __noinline__ uint32_t largest_key(const uint64_t *cand, const int *s_cnt, uint32_t *s_mm, uint32_t top)
{
    __syncthreads();                 // the candidates are listed
    const int tid = threadIdx.x, cnt = min(*s_cnt, RANK_MAX);
    uint32_t hi = 0u;
    for (int c = tid; c < cnt; c += TT) hi = max(hi, (uint32_t)(cand[c] >> 32));
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((tid & 31) == 0) s_mm[tid >> 5] = hi;
    __syncthreads();
    for (int w = 0; w < TT / 32; ++w) top = max(top, s_mm[w]);
    return top;
}

// Shared memory of one CTA of the block-level select.
struct ThreshSmem {
    uint32_t *ukeys;        // staged group maxima or a short row (dynamic)
    uint64_t *cand;         // CAP candidate words
    uint32_t *hist;         // the bins, then the list of qualifying groups (GLIST words)
    uint32_t *wsum, *s3;
    int *s_cnt, *s_ng, *s_misc;
    uint32_t *s_mm;
    uint64_t *sorted;       // RANK_MAX words, in the keys' place once the candidates are listed
};

// The block-level select of row i of piece pc (ends with the row written; the
// caller separates rows by a barrier).
__device__ __forceinline__ void thresh_row(const float *__restrict__ S, const float *__restrict__ tops,
                                           const Piece &pc, int i, int32_t *__restrict__ tsel_idx, float *__restrict__ tsel_cos,
                                           int32_t stride_t, int32_t *__restrict__ lsel_idx,
                                           float *__restrict__ lsel_cos, int32_t stride_l,
                                           int32_t *__restrict__ n_fallback, const ThreshSmem &sm)
{
    uint32_t *ukeys = sm.ukeys, *hist = sm.hist, *wsum = sm.wsum, *s3 = sm.s3;
    uint64_t *cand = sm.cand;
    int &s_cnt = *sm.s_cnt, &s_ng = *sm.s_ng;
    int *s_misc = sm.s_misc;

    const int tid = threadIdx.x;
    const bool is_tgt = i < pc.ntr;
    const int R = is_tgt ? pc.keep_t : pc.keep_l;
    int32_t *oi;
    float *oc;
    int stride;
    if (is_tgt) {
        const int64_t o = (pc.t_row0 + i) * (int64_t)stride_t;
        oi = tsel_idx + o;
        oc = tsel_cos ? tsel_cos + o : nullptr;
        stride = stride_t;
    } else {
        const int64_t o = (pc.l_row0 + (i - pc.ntr)) * (int64_t)stride_l;
        oi = lsel_idx + o;
        oc = lsel_cos ? lsel_cos + o : nullptr;
        stride = stride_l;
    }
    const int n = pc.n;
    const float *row = S + pc.s_off + (int64_t)i * pc.ld;
    const int gshift = pc.gshift;
    const int64_t n_groups = group_count(n, gshift);
    const int U = (int)min(n_groups, (int64_t)UNION_MAX);
    if (tid == 0) { s_cnt = 0; s_ng = 0; }
    uint32_t T = 0u, top = 0xffffffffu;    // the candidates' keys lie in [T, top]

    // For tau = key_value(T) and non-NaN x,
    // x >= tau holds exactly when order_key(x) >= T, so the passes below
    // compare floats and build keys only for the entries they keep.  (T lies
    // between two keys of the row, so tau is a number, and -0 only for a T
    // that both zeros' key reaches.)
    if (U >= R) {
        // (tau at most the R-th largest of the group maxima: a few groups more
        // cost less than the last bits of the search); then the groups whose
        // maximum reaches it, in any order
        const float *tp = tops + pc.tops_off + (int64_t)i * group_stride(n, gshift);
        for (int j = tid; j < U; j += TT) ukeys[j] = order_key(__ldg(tp + j));
        T = kth_lower(ukeys, U, R, R / 8 + 8, hist, wsum, s3, sm.s_mm, top);
        const float tau = key_value(T);
        for (int j = tid; j < U; j += TT) {
            if (ukeys[j] >= T) {
                const int pos = atomicAdd(&s_ng, 1);
                if (pos < GLIST) hist[pos] = (uint32_t)j;
            }
        }
        __syncthreads();
        const int ng = s_ng;
        if (ng <= GLIST) {
            // the qualifying groups, read as float4 slots (a group of 32 is
            // eight slots, of 8 two); group starts are 32-byte aligned and a
            // row holds round_up(n, 32) floats, so a slot never leaves it
            const int sshift = gshift - 2;
            const int smask = (1 << sshift) - 1;
            const int slots = ng << sshift;
            for (int s0 = 0; s0 < slots; s0 += TT * UNROLL) {
                float4 v[UNROLL];
                int j4[UNROLL];
#pragma unroll
                for (int u = 0; u < UNROLL; ++u) {
                    const int sl = s0 + u * TT + tid;
                    j4[u] = sl < slots ? (int)((hist[sl >> sshift] << gshift) + ((sl & smask) << 2)) : n;
                    v[u] = j4[u] < n ? __ldcs(reinterpret_cast<const float4 *>(row + j4[u]))
                                     : make_float4(-1e30f, -1e30f, -1e30f, -1e30f);
                }
#pragma unroll
                for (int u = 0; u < UNROLL; ++u) {
                    if (j4[u] >= n) continue;
                    const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (j4[u] + c < n && x[c] >= tau) push_cand(cand, &s_cnt, x[c], j4[u] + c);
                }
            }
            // groups past the staged union (rows of more than 8,192 groups)
            if (n_groups > U) stream_tail(row, U << gshift, n, tau, cand, &s_cnt);
        } else {
            stream_tail(row, 0, n, tau, cand, &s_cnt);
        }
        if (n_groups > U) top = largest_key(cand, &s_cnt, sm.s_mm, top);
    } else if (n <= kSelectSortAll) {
        // a short row: every entry staged, its R-th largest key found in shared memory
        for (int j = tid; j < n; j += TT) ukeys[j] = order_key(__ldcs(row + j));
        T = kth_lower(ukeys, n, R, R / 8 + 8, hist, wsum, s3, sm.s_mm, top);
        for (int j = tid; j < n; j += TT) {
            const uint32_t k = ukeys[j];
            if (k >= T) {
                const int pos = atomicAdd(&s_cnt, 1);
                if (pos < CAP) cand[pos] = cand_word(k, j);
            }
        }
    } else {
        // (the planner sends no such row; every entry is a candidate, and the
        // exact select below stands in when they overflow the buffer)
        __syncthreads();
        stream_tail(row, 0, n, -__int_as_float(0x7f800000), cand, &s_cnt);
    }
    __syncthreads();
    const int cnt = s_cnt;
    // (fewer than R candidates cannot happen with group maxima of this row;
    // the exact select then stands in rather than list unfilled entries)
    if (cnt >= R && cnt <= RANK_MAX) {
        rank_words(cand, cnt, R, T, top, hist, wsum, sm.sorted, oi, oc);
        for (int c = R + tid; c < stride; c += TT) {
            oi[c] = -1;
            if (oc) oc[c] = 0.f;
        }
    } else if (cnt >= R && cnt <= CAP) {
        int P = 1;
        while (P < cnt) P <<= 1;
        for (int j = cnt + tid; j < P; j += TT) cand[j] = 0ull;
        __syncthreads();
        bitonic_desc<TT>(cand, P);
        write_list<TT>(cand, R, 0, nullptr, oi, oc, stride, 0.f);
    } else {
        if (tid == 0) atomicAdd(n_fallback, 1);
        select_row_global<TT>(row, n, R, cand, hist, s_misc, oi, oc, stride, 0.f);
    }
}

#define THRESH_SMEM                                   \
    extern __shared__ __align__(8) uint32_t ukeys[];  \
    __shared__ uint64_t cand[CAP];                    \
    __shared__ uint32_t hist[GLIST];                  \
    __shared__ uint32_t wsum[TT / 32];                \
    __shared__ uint32_t s3[3];                        \
    __shared__ int s_cnt, s_ng;                       \
    __shared__ int s_misc[TT / 32 + 3];               \
    __shared__ uint32_t s_mm[TT / 16];                \
    static_assert(BINS <= GLIST && RANK_MAX * 8 <= kSelectSortAll * 4, "shared arrays reused"); \
    const ThreshSmem sm{ukeys, cand, hist, wsum, s3, &s_cnt, &s_ng, s_misc, s_mm,               \
                        reinterpret_cast<uint64_t *>(ukeys)};

// One CTA per row of the pieces' general rows.
__global__ void __launch_bounds__(TT, 6)
select_thresh_kernel(const float *__restrict__ S, const float *__restrict__ tops, const Piece *__restrict__ pieces,
                     int32_t n_pieces, int32_t *__restrict__ tsel_idx, float *__restrict__ tsel_cos, int32_t stride_t,
                     int32_t *__restrict__ lsel_idx, float *__restrict__ lsel_cos, int32_t stride_l,
                     int32_t *__restrict__ n_fallback)
{
    THRESH_SMEM
    const Piece pc = pieces[find_piece(pieces, n_pieces, blockIdx.x, [](const Piece &x) { return x.gblock_begin; })];
    thresh_row(S, tops, pc, pc.g0 + (int)(blockIdx.x - pc.gblock_begin), tsel_idx, tsel_cos, stride_t, lsel_idx,
               lsel_cos, stride_l, n_fallback, sm);
}

// The rows the warp-level select handed on (row_list[0] of them, listed
// from row_list[1]), a grid-stride loop of CTAs.
__global__ void __launch_bounds__(TT)
select_thresh_list_kernel(const float *__restrict__ S, const float *__restrict__ tops,
                          const Piece *__restrict__ pieces, int32_t n_pieces, int32_t *__restrict__ tsel_idx,
                          float *__restrict__ tsel_cos, int32_t stride_t, int32_t *__restrict__ lsel_idx,
                          float *__restrict__ lsel_cos, int32_t stride_l, int32_t *__restrict__ n_fallback,
                          const int32_t *__restrict__ row_list)
{
    THRESH_SMEM
    const int count = row_list[0];
    for (int k = blockIdx.x; k < count; k += gridDim.x) {
        const int64_t b = row_list[1 + k];
        const Piece pc = pieces[find_piece(pieces, n_pieces, b, [](const Piece &x) { return x.tblock_begin; })];
        thresh_row(S, tops, pc, pc.th0 + (int)(b - pc.tblock_begin), tsel_idx, tsel_cos, stride_t, lsel_idx, lsel_cos,
                   stride_l, n_fallback, sm);
        __syncthreads();            // the next row reuses the shared arrays
    }
}

// ---------------------------------------------------------------------------
// Warp-level select of the rows of small scenes (groups of 8 objects) with
// lists of at most NARROW_R entries, in launches of many rows: one warp per
// row, no block barriers, the group maxima as keys (at most 1,024; or, for a
// row with fewer group maxima than its list length, at most 1,024 entries,
// ranked directly).
// A bound T of the R-th largest key is found by value bins, the groups whose
// maximum reaches it are gathered, and the candidates are ranked by value bins
// (their words are all distinct).  A row whose groups or candidates overflow
// the warp's buffers is appended to row_list for the block-level select.
// Instruction issue bounds it (83% of the slots with a bitwise search over 32
// keys per lane whatever the row's length, and ranks by counting).
// On the 67-scene batch, whose many small scenes' lists of 95 and 16 entries
// these are: 0.28 ms, against 0.68 with those and 1.02 with a CTA per row.
constexpr int WS_KEYS = 1024;   // keys per row
constexpr int WS_CAP = 256;     // candidate words per warp
constexpr int WW = 8;           // warps (rows) per CTA
constexpr int WS_GL = 320;      // qualifying groups per warp
constexpr int NARROW_R = 128;   // longest list

// The keys of a row held by a warp, KPL per lane: the bound T and the groups
// (or entries) reaching it.
template <int KPL, class Load, class Take>
__device__ __forceinline__ uint32_t warp_bound(int U, int R, uint32_t *hist, int lane, uint32_t &top, Load load, Take take)
{
    uint32_t key[KPL], lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        const int g = lane + 32 * k;
        key[k] = g < U ? load(g) : 0u;       // 0: no value
        if (g < U) {
            lo = min(lo, key[k]);
            hi = max(hi, key[k]);
        }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    top = __reduce_max_sync(0xffffffffu, hi);
    uint32_t base = lo, span = top - lo, rank = (uint32_t)R;
    const uint32_t slack = (uint32_t)R / 8u + 4u;
#pragma unroll 1
    for (;;) {
        const int shift = bin_shift(span);
        warp_clear_bins(hist, lane);
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            const uint32_t d = key[k] - base;
            if (lane + 32 * k < U && key[k] >= base && d <= span) atomicAdd(&hist[bin_slot(d >> shift)], 1u);
        }
        __syncwarp();
        uint32_t rem, cnt;
        const uint32_t b = warp_find_bin(hist, rank, lane, rem, cnt);
        __syncwarp();
        base += b << shift;
        if (shift == 0 || cnt - rem <= slack) break;
        span = min(span - (b << shift), (1u << shift) - 1u);
        rank = rem;
    }
#pragma unroll
    for (int k = 0; k < KPL; ++k)
        if (32 * k < U) take(lane + 32 * k < U && key[k] >= base, key[k], lane + 32 * k);
    return base;
}

__global__ void __launch_bounds__(WW * 32, 4)
select_warp_small_kernel(const float *__restrict__ S, const float *__restrict__ tops, const Piece *__restrict__ pieces,
                         int32_t n_pieces, int64_t total_rows, int32_t *__restrict__ tsel_idx,
                         float *__restrict__ tsel_cos, int32_t stride_t, int32_t *__restrict__ lsel_idx,
                         float *__restrict__ lsel_cos, int32_t stride_l, int32_t *__restrict__ row_list)
{
    __shared__ uint32_t hist_all[WW][WS_GL];      // the bins; between their two uses the list of groups
    __shared__ uint64_t cand_all[WW][2 * WS_CAP]; // the candidates, then their layout by bins
    static_assert(WS_GL >= kWarpBins, "the group list and the bins share their place");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t = (int64_t)blockIdx.x * WW + warp;
    if (t >= total_rows) return;            // (warp-uniform)
    uint32_t *hist = hist_all[warp], *glist = hist;
    uint64_t *cand = cand_all[warp];
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u;
    auto hand_on = [&]() {
        if (lane == 0) row_list[1 + atomicAdd(&row_list[0], 1)] = (int32_t)t;
    };
    // the piece of thresholded row t (the last whose tblock_begin <= t)
    int lo = 0, hi = n_pieces - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pieces[mid].tblock_begin <= t) lo = mid;
        else hi = mid - 1;
    }
    const Piece &pc = pieces[lo];
    const int i = pc.th0 + (int)(t - pc.tblock_begin);
    const bool is_tgt = i < pc.ntr;
    const int R = is_tgt ? pc.keep_t : pc.keep_l;
    const int n = pc.n;
    const int gshift = pc.gshift;
    const int64_t n_groups = group_count(n, gshift);
    // a row with fewer group maxima than R (a short row), or not many more (whose
    // R-th largest maximum would let half the row through), ranks its entries
    // themselves: a bound of their R-th largest key, then every entry reaching it
    const bool entries = n_groups < R || (n <= WS_KEYS && 2 * n_groups < 3 * R);
    if (gshift != kGroupShiftSmall || R > NARROW_R || (entries ? (int64_t)n : n_groups) > WS_KEYS)
        return;    // the block-level select's row
    const int U = entries ? n : (int)n_groups;
    const float *row = S + pc.s_off + (int64_t)i * pc.ld;
    const float *tp = tops + pc.tops_off + (int64_t)i * group_stride(n, gshift);
    uint32_t T, top;
    int cnt = 0, ng = 0;
    auto load = [&](int g) { return order_key(entries ? __ldcs(row + g) : __ldg(tp + g)); };
    auto take = [&](bool q, uint32_t k, int g) {
        const unsigned bal = __ballot_sync(FULL, q);
        if (entries) {
            if (q) {
                const int pos = cnt + __popc(bal & lt);
                if (pos < WS_CAP) cand[pos] = cand_word(k, g);
            }
            cnt += __popc(bal);
        } else {
            if (q) {
                const int pos = ng + __popc(bal & lt);
                if (pos < WS_GL) glist[pos] = (uint32_t)g;
            }
            ng += __popc(bal);
        }
    };
    if (U <= 128) T = warp_bound<4>(U, R, hist, lane, top, load, take);
    else if (U <= 256) T = warp_bound<8>(U, R, hist, lane, top, load, take);
    else if (U <= 512) T = warp_bound<16>(U, R, hist, lane, top, load, take);
    else T = warp_bound<32>(U, R, hist, lane, top, load, take);
    if (!entries) {
        if (ng > WS_GL) { hand_on(); return; }
        __syncwarp();
        // the groups' entries >= tau, read as float4 slots (two to a group of
        // 8; group starts are 32-byte aligned and a row holds round_up(n, 32)
        // floats, so a slot never leaves it)
        const float tau = key_value(T);
        const int slots = 2 * ng;
        for (int s0 = 0; s0 < slots; s0 += 32 * 4) {
            float4 v[4];
            int j4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int sl = s0 + 32 * u + lane;
                j4[u] = sl < slots ? (int)((glist[sl >> 1] << 3) + ((sl & 1) << 2)) : n;
                v[u] = j4[u] < n ? __ldcs(reinterpret_cast<const float4 *>(row + j4[u])) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (s0 + 32 * u >= slots) break;     // (warp-uniform: short lists take few ballots)
                const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const bool q = j4[u] + c < n && x[c] >= tau;
                    const unsigned bal = __ballot_sync(FULL, q);
                    if (q) {
                        const int pos = cnt + __popc(bal & lt);
                        if (pos < WS_CAP) cand[pos] = cand_word(order_key(x[c]), j4[u] + c);
                    }
                    cnt += __popc(bal);
                }
            }
        }
    }
    if (cnt > WS_CAP || cnt < R) { hand_on(); return; }
    __syncwarp();
    int32_t *oi;
    float *oc;
    int stride;
    if (is_tgt) {
        const int64_t o = (pc.t_row0 + i) * (int64_t)stride_t;
        oi = tsel_idx + o;
        oc = tsel_cos ? tsel_cos + o : nullptr;
        stride = stride_t;
    } else {
        const int64_t o = (pc.l_row0 + (i - pc.ntr)) * (int64_t)stride_l;
        oi = lsel_idx + o;
        oc = lsel_cos ? lsel_cos + o : nullptr;
        stride = stride_l;
    }
    warp_rank_words(cand, cnt, R, T, top, hist, cand + WS_CAP, lane, [&](uint64_t w, int r) {
        oi[r] = (int32_t)(0xffffffffu - (uint32_t)(w & 0xffffffffu));
        if (oc) oc[r] = key_value((uint32_t)(w >> 32));
    });
    for (int k = R + lane; k < stride; k += 32) {
        oi[k] = -1;
        if (oc) oc[k] = 0.f;
    }
}

}  // namespace

// Rows of launches of at most this many take a CTA per row whatever their
// kind: the warps of the small-row kernel would leave most of the chip idle
// and each run its whole chain of searches and loads alone (one query in a
// 200-object scene: 6.5 us against 15 for the small-row kernel and its list).
constexpr int64_t kBlockRows = 1216;

void select_general_rows(Piece *pieces, size_t n, int64_t total_rows, int64_t *general, bool *small)
{
    auto small_kind = [](const Piece &p, int32_t keep) {
        const int64_t g = group_count(p.n, p.gshift);
        return p.gshift == kGroupShiftSmall && keep <= NARROW_R && (g < keep ? (int64_t)p.n : g) <= WS_KEYS;
    };
    *general = 0;
    *small = false;
    for (size_t k = 0; k < n; ++k) {
        Piece &p = pieces[k];
        // target rows [th0, ntr), landmark rows [max(th0, ntr), rows)
        const int32_t t1 = p.th0 < p.ntr ? p.ntr : p.th0;
        const bool st = total_rows > kBlockRows && small_kind(p, p.keep_t);
        const bool sl = total_rows > kBlockRows && small_kind(p, p.keep_l);
        *small |= (st && p.th0 < t1) || (sl && t1 < p.rows);
        p.g0 = st ? t1 : p.th0;
        const int32_t g1 = sl ? t1 : p.rows;
        p.gblock_begin = *general;
        *general += g1 > p.g0 ? g1 - p.g0 : 0;
    }
}

cudaError_t launch_select_thresh(const float *S, const float *tops, const Piece *pieces, int32_t n_pieces,
                                 int64_t total_rows, int64_t general, bool small, int32_t max_union,
                                 int32_t *tsel_idx, float *tsel_cos, int32_t stride_t, int32_t *lsel_idx,
                                 float *lsel_cos, int32_t stride_l, int32_t *n_fallback, int32_t *row_list,
                                 cudaStream_t s)
{
    if (total_rows <= 0) return cudaSuccess;
    if (n_pieces < 1 || total_rows > 0x7fffffff || max_union < 1 || ((uintptr_t)S & 15u) != 0 ||
        ((uintptr_t)tops & 15u) != 0 || !n_fallback || (small && !row_list))
        return cudaErrorInvalidValue;
    // the staged group maxima, or a whole short row
    const int32_t staged = max_union < UNION_MAX ? (max_union > kSelectSortAll ? max_union : kSelectSortAll) : UNION_MAX;
    const size_t smem = (size_t)staged * sizeof(uint32_t);
    static_assert(CAP >= kSelectSortAll, "rows that take every entry fit the candidate buffer");
    cudaError_t e;
    if (general > 0) {
        e = cudaFuncSetAttribute(select_thresh_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        select_thresh_kernel<<<(unsigned)general, TT, smem, s>>>(S, tops, pieces, n_pieces, tsel_idx, tsel_cos,
                                                                 stride_t, lsel_idx, lsel_cos, stride_l, n_fallback);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (!small) return cudaSuccess;
    // the small rows, then those they hand on
    if ((e = cudaMemsetAsync(row_list, 0, sizeof(int32_t), s)) != cudaSuccess) return e;
    select_warp_small_kernel<<<(unsigned)((total_rows + WW - 1) / WW), WW * 32, 0, s>>>(
        S, tops, pieces, n_pieces, total_rows, tsel_idx, tsel_cos, stride_t, lsel_idx, lsel_cos, stride_l, row_list);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(select_thresh_list_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t grid = total_rows < 304 ? total_rows : 304;
    select_thresh_list_kernel<<<(unsigned)grid, TT, smem, s>>>(S, tops, pieces, n_pieces, tsel_idx, tsel_cos,
                                                               stride_t, lsel_idx, lsel_cos, stride_l, n_fallback,
                                                               row_list);
    return cudaGetLastError();
}

}  // namespace farm
