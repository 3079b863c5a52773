// k_sim_few.cu -- FP32-accurate descriptor similarity for few query rows
// (App. D.2 step 3 for one question, or a handful): at most kSimFewRows rows
// per block against every object of its scene.
//
// What bounds such a product is reading the descriptors (92 MB of FP16 parts at
// 20,000 objects, D = 1152), so the work is split over objects as finely as
// the tensor cores allow and nothing is spent on padding the query rows: the
// roles of the operands are exchanged, 128 objects are the rows (M) of the MMA
// and the query rows, padded to 16, 32, 64 or 128, its columns (N).  157 CTAs
// of 128 objects cover a 20,000-object scene, two to an SM, against 79 tiles
// of 256 objects in the kernels of k_sim_tc.cu, which also multiply up to 128
// rows of padding.  Each product of a cosine is the same, and the sums run in
// the same K order into the same two accumulators (hi.hi; hi.lo then lo.hi per
// K step of 16), so cosines are bitwise those kernels'.
//
// Measured at 20,000 objects, D = 1152: 48 rows (farm_rank_rows_noalloc with its
// normalisation and select, descriptors in L2) 19.7 us a call against 44.3 with
// CTA pairs; 12 queries of 42 rows (farm_query_batch) 192 us against 234, its
// similarity 29 us from cold caches against 70 for the fused selection's two
// launches.  The line lies at 128 rows, one M tile of the other kernels: above
// it they pad no more than this one and read each descriptor once per 128 or
// 256 rows just the same.
//
// Per CTA (192 threads): warp 0 issues the TMA loads of each K slice (32 FP16
// values of four tiles d_hi, d_lo, q_hi, q_lo, 64-byte swizzle), one thread of
// warp 1 the MMAs, warps 2-5 drain TMEM: a lane holds one object, so the store
// of a query row's 32 cosines is one 128-byte line, and the maximum of a group
// of objects a reduction over lanes.  Every wait is bounded.
#include <type_traits>

#include "tc_common.cuh"

namespace farm {
namespace {

using namespace tc;
using E = Elem<kSimF16x3>;

constexpr int BO = 128;                 // objects per CTA
constexpr int TH = 192;

template <int NQ>
struct FewCfg {
    static constexpr int D_BYTES = BO * E::ROW_BYTES;              // one part of the objects' slice
    static constexpr int Q_BYTES = NQ * E::ROW_BYTES;
    static constexpr int STAGE_BYTES = 2 * (D_BYTES + Q_BYTES);
    static constexpr int STAGES = 110 * 1024 / STAGE_BYTES < 8 ? 110 * 1024 / STAGE_BYTES : 8;   // two CTAs per SM
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
    static constexpr uint32_t TMEM_COLS = 2 * NQ < 32 ? 32 : 2 * NQ;   // main and correction accumulators
    static_assert(Q_BYTES % 512 == 0 && SMEM_BYTES <= 113 * 1024 && STAGES >= 3 && TMEM_COLS <= 256, "few-row tile");
};

__device__ __forceinline__ void mma_few(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t id,
                                        uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(id), "r"(accumulate));
}

// 16 columns of the warp's 32 TMEM lanes, without the wait.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

template <int NQ, bool GROUPED>
__global__ void __launch_bounds__(TH, 2)
sim_few_kernel(const __grid_constant__ CUtensorMap map_q0, const __grid_constant__ CUtensorMap map_q1,
               const __grid_constant__ CUtensorMap map_d0, const __grid_constant__ CUtensorMap map_d1,
               const GemmPiece *__restrict__ pieces, int32_t n_pieces, const GemmPiece single, float *__restrict__ S,
               float *__restrict__ tops, int32_t k_slices, int32_t *err)
{
    using C = FewCfg<NQ>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::STAGES * C::STAGE_BYTES);
    uint64_t *empty = full + C::STAGES;
    uint64_t *acc_full = empty + C::STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(acc_full, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(C::TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    const int tile = blockIdx.x;
    const GemmPiece pc = piece_of<GROUPED>(tile, pieces, n_pieces, single);
    const int n0 = (tile - pc.tile_begin) * BO;

    if (warp == 0) {
        if (lane == 0) {
            const CUtensorMap *d0 = GROUPED ? static_cast<const CUtensorMap *>(pc.bmap) : &map_d0;
            const CUtensorMap *d1 = GROUPED ? static_cast<const CUtensorMap *>(pc.bmap) + 1 : &map_d1;
            int kb = 0;
            if (GROUPED && (reinterpret_cast<uintptr_t>(pc.bmap) & 63u)) {
                // a tensor map must be 64-byte aligned: never hand the copy engine anything else
                atomicOr(err, kErrPieceTable);
                *abort_flag = 1;
            }
            for (; kb < k_slices && !*abort_flag; ++kb) {
                const int s = kb % C::STAGES;
                if (!mbar_wait(&empty[s], ((kb / C::STAGES) & 1u) ^ 1u) || *abort_flag) {
                    *abort_flag = 1;
                    break;
                }
                uint8_t *st = smem + s * C::STAGE_BYTES;
                const int kx = kb * E::BK;
                mbar_expect_tx(&full[s], C::STAGE_BYTES);
                tma_load_2d(st, d0, &full[s], kx, n0);
                tma_load_2d(st + C::D_BYTES, d1, &full[s], kx, n0);
                tma_load_2d(st + 2 * C::D_BYTES, &map_q0, &full[s], kx, (int)pc.q_row0);
                tma_load_2d(st + 2 * C::D_BYTES + C::Q_BYTES, &map_q1, &full[s], kx, (int)pc.q_row0);
            }
            if (*abort_flag) {
                // let the copies already issued land before shared memory is released
                for (int j = kb > C::STAGES ? kb - C::STAGES : 0; j < kb; ++j)
                    mbar_wait(&full[j % C::STAGES], (j / C::STAGES) & 1u);
                atomicOr(err, kErrTimeout);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t id = idesc(0u, NQ, BO);
            for (int kb = 0; kb < k_slices; ++kb) {
                const int s = kb % C::STAGES;
                if (!mbar_wait(&full[s], (kb / C::STAGES) & 1u) || *abort_flag) {
                    *abort_flag = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t d_hi = smem_u32(smem + s * C::STAGE_BYTES), d_lo = d_hi + C::D_BYTES;
                const uint32_t q_hi = d_hi + 2 * C::D_BYTES, q_lo = q_hi + C::Q_BYTES;
#pragma unroll
                for (int kk = 0; kk < E::KSTEPS; ++kk) {
                    const uint32_t off = kk * 32;     // 16 FP16 values = 32 bytes along K
                    const uint32_t first = (kb | kk) != 0;
                    mma_few(tmem, smem_desc<kSimF16x3>(d_hi + off), smem_desc<kSimF16x3>(q_hi + off), id, first);
                    mma_few(tmem + NQ, smem_desc<kSimF16x3>(d_lo + off), smem_desc<kSimF16x3>(q_hi + off), id, first);
                    mma_few(tmem + NQ, smem_desc<kSimF16x3>(d_hi + off), smem_desc<kSimF16x3>(q_lo + off), id, 1u);
                }
                mma_commit(&empty[s]);
            }
            if (!*abort_flag) mma_commit(acc_full);
            else atomicOr(err, kErrTimeout);
        }
    } else {
        const int quad = warp & 3;
        const int64_t j0 = (int64_t)n0 + quad * 32, j = j0 + lane, n = pc.n;
        const int64_t gs = group_stride(n, pc.gshift);
        const bool keep_tops = tops != nullptr && pc.tops_off >= 0;
        float *out = S + pc.s_off + j;
        float *top = tops + (keep_tops ? pc.tops_off + (j >> pc.gshift) : 0);
        if (!mbar_wait(acc_full, 0u) || *abort_flag) {
            *abort_flag = 1;
        } else {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
            for (int c = 0; c < NQ && c < pc.rows; c += 16) {
                uint32_t a[16], b[16];
                tmem_ld16_issue(tb + (uint32_t)c, a);
                tmem_ld16_issue(tb + NQ + (uint32_t)c, b);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int r = c + i;
                    if (r >= pc.rows) break;                     // (warp-uniform)
                    const float v = fmaf(__uint_as_float(b[i]), RESID_SCALE_INV, __uint_as_float(a[i]));
                    if (j < n) out[(int64_t)r * pc.ld] = v;
                    if (!keep_tops) continue;
                    // the group's maximum (-inf when it lies past the row's end)
                    if (pc.gshift == kGroupShift) {
                        const uint32_t k = __reduce_max_sync(0xffffffffu, j < n ? order_key(v) : 0x007fffffu);
                        if (lane == 0) top[r * gs] = key_value(k);
                    } else {
                        float m = j < n ? v : -__int_as_float(0x7f800000);
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                        if ((lane & 7) == 0) top[r * gs] = m;
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS));
    }
}

template <int NQ, bool GROUPED>
cudaError_t launch_nq(const uint16_t *q_hi, const uint16_t *q_lo, int64_t rows_total, const CUtensorMap *d0,
                      const CUtensorMap *d1, int32_t dim_pad, const GemmPiece *pieces, int32_t n_pieces,
                      const GemmPiece &single, int64_t tiles, float *S, float *tops, int32_t *err, cudaStream_t s)
{
    using C = FewCfg<NQ>;
    CUtensorMap mq0, mq1;
    if (!make_map<kSimF16x3>(&mq0, q_hi, dim_pad, rows_total, NQ) || !make_map<kSimF16x3>(&mq1, q_lo, dim_pad, rows_total, NQ))
        return cudaErrorInvalidValue;
    auto kernel = sim_few_kernel<NQ, GROUPED>;
    static bool ready[64] = {};          // per device: the attribute is set (concurrent first calls set the same)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !ready[dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) ready[dev] = true;
    }
    kernel<<<(unsigned)tiles, TH, C::SMEM_BYTES, s>>>(mq0, mq1, d0 ? *d0 : mq0, d1 ? *d1 : mq1, pieces, n_pieces, single,
                                                      S, tops, (dim_pad + E::BK - 1) / E::BK, err);
    return cudaGetLastError();
}

template <bool GROUPED>
cudaError_t launch_rows(int64_t rows, const uint16_t *q_hi, const uint16_t *q_lo, int64_t rows_total,
                        const CUtensorMap *d0, const CUtensorMap *d1, int32_t dim_pad, const GemmPiece *pieces,
                        int32_t n_pieces, const GemmPiece &single, int64_t tiles, float *S, float *tops, int32_t *err,
                        cudaStream_t s)
{
    if (tiles <= 0) return cudaSuccess;
    if (rows < 1 || rows > kSimFewRows || tiles > 0x7fffffffLL || rows_total > 0x7fffffffLL || dim_pad % kDimAlign != 0)
        return cudaErrorInvalidValue;
    if (!get_encoder()) return cudaErrorNotSupported;
    if (((uintptr_t)q_hi | (uintptr_t)q_lo) & 15u) return cudaErrorMisalignedAddress;
    auto go = [&](auto nq) {
        return launch_nq<decltype(nq)::value, GROUPED>(q_hi, q_lo, rows_total, d0, d1, dim_pad, pieces, n_pieces, single,
                                                       tiles, S, tops, err, s);
    };
    if (rows <= 16) return go(std::integral_constant<int, 16>{});
    if (rows <= 32) return go(std::integral_constant<int, 32>{});
    if (rows <= 64) return go(std::integral_constant<int, 64>{});
    return go(std::integral_constant<int, 128>{});
}

}  // namespace

cudaError_t launch_sim_few(const uint16_t *q_hi, const uint16_t *q_lo, const uint16_t *d_hi, const uint16_t *d_lo,
                           float *S, int64_t rows, int64_t n, int32_t dim_pad, int64_t ld_s, float *tops, int32_t *err,
                           cudaStream_t s)
{
    if (rows <= 0 || n <= 0) return cudaSuccess;
    if (n > 0x7fffffffLL || ld_s < n || ld_s > 0x7fffffffLL || dim_pad % kDimAlign != 0) return cudaErrorInvalidValue;
    if (!get_encoder()) return cudaErrorNotSupported;
    if (((uintptr_t)d_hi | (uintptr_t)d_lo | (tops ? (uintptr_t)tops : 0)) & 15u) return cudaErrorMisalignedAddress;
    CUtensorMap d0, d1;
    if (!make_map<kSimF16x3>(&d0, d_hi, dim_pad, n, BO) || !make_map<kSimF16x3>(&d1, d_lo, dim_pad, n, BO))
        return cudaErrorInvalidValue;
    GemmPiece p{};
    p.tops_off = tops ? 0 : -1;
    p.rows = (int32_t)rows;
    p.n = p.n_store = (int32_t)n;
    p.ld = (int32_t)ld_s;
    p.gshift = group_shift_for(n);
    p.col_mode = kColAll;
    return launch_rows<false>(rows, q_hi, q_lo, rows, &d0, &d1, dim_pad, nullptr, 1, p, (n + BO - 1) / BO, S, tops, err, s);
}

cudaError_t launch_sim_few_grouped(const uint16_t *q_hi, const uint16_t *q_lo, int64_t rows_total, int32_t dim_pad,
                                   const GemmPiece *pieces, int32_t n_pieces, int64_t total_tiles, float *S,
                                   float *tops, int32_t *err, cudaStream_t s)
{
    if (n_pieces < 1 || !pieces) return cudaErrorInvalidValue;
    // (a piece holds at most kSimFewRows rows and at most rows_total)
    return launch_rows<true>(rows_total < kSimFewRows ? rows_total : kSimFewRows, q_hi, q_lo, rows_total, nullptr, nullptr,
                             dim_pad, pieces, n_pieces, GemmPiece{}, total_tiles, S, tops, err, s);
}

cudaError_t preload_sim_few()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, sim_few_kernel<16, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, sim_few_kernel<32, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, sim_few_kernel<64, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, sim_few_kernel<128, false>);
    return e;
}

}  // namespace farm
