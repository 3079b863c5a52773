// tc_common.cuh -- what the tensor-core similarity kernels (k_sim_tc.cu,
// k_sim_few.cu) share: mbarriers with bounded waits, TMA loads, TMEM loads,
// shared-memory and instruction descriptors, tensor maps.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include "farm_internal.h"

namespace farm {
namespace tc {

constexpr uint32_t WAIT_LIMIT = 1u << 24;    // try_wait polls before giving up (about a second)
constexpr float RESID_SCALE_INV = 1.f / 2048.f;   // the residual operands carry a factor 2^11

// Per-mode element layout of the operand rows of a K slice.
template <int MODE>
struct Elem;
template <>
struct Elem<kSimF16x3> {                     // three-term FP16 with scaled residuals
    static constexpr int BK = 32;            // FP16 elements per K slice (64-byte rows)
    static constexpr int ROW_BYTES = 64;
    static constexpr int KSTEPS = 2;         // 16 FP16 values (32 bytes) per MMA
    static constexpr bool SPLIT = true;      // hi and lo tiles of each operand
    static constexpr uint64_t LAYOUT = 4;    // 64-byte swizzle
    static constexpr uint32_t SBO = 512;     // 8 rows x 64 bytes
};
template <>
struct Elem<kSimBf16> {                      // BF16
    static constexpr int BK = 64;            // BF16 elements per K slice (128-byte rows)
    static constexpr int ROW_BYTES = 128;
    static constexpr int KSTEPS = 4;         // 16 BF16 values (32 bytes) per MMA
    static constexpr bool SPLIT = false;
    static constexpr uint64_t LAYOUT = 2;    // 128-byte swizzle
    static constexpr uint32_t SBO = 1024;    // 8 rows x 128 bytes
};
template <>
struct Elem<kSimFp8> {                       // FP8 E4M3
    static constexpr int BK = 128;           // FP8 elements per K slice (128-byte rows)
    static constexpr int ROW_BYTES = 128;
    static constexpr int KSTEPS = 4;         // 32 FP8 values (32 bytes) per MMA
    static constexpr bool SPLIT = false;
    static constexpr uint64_t LAYOUT = 2;    // 128-byte swizzle
    static constexpr uint32_t SBO = 1024;    // 8 rows x 128 bytes
};

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// Bounded wait for the phase with the given parity; false on expiry.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    const uint32_t a = smem_u32(bar);
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// One non-blocking test of the phase with the given parity.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile with rows of
// ROW_BYTES swizzled in 8-row core groups SBO bytes apart; version 1.  The
// leading byte offset is unused for swizzled K-major layouts.
template <int MODE>
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);              // start address
    d |= (uint64_t)(Elem<MODE>::SBO >> 4) << 32;            // stride byte offset
    d |= (uint64_t)1 << 46;                                 // descriptor version
    d |= Elem<MODE>::LAYOUT << 61;                          // swizzle mode
    return d;
}

// Instruction descriptors: D = F32, A and B K-major, M = m (128, or 256 for
// a CTA pair), N = n; operand format FP16 (0, kind::f16), BF16 (1,
// kind::f16) or E4M3 (0, kind::f8f6f4).
__host__ __device__ constexpr uint32_t idesc(uint32_t ab_format, int n, int m)
{
    return (1u << 4)                      // D format F32
           | (ab_format << 7)             // A format
           | (ab_format << 10)            // B format
           | ((uint32_t)(n >> 3) << 17)   // N / 8
           | ((uint32_t)(m >> 4) << 24);  // M / 16
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ uint32_t order_key(float f)
{
    const uint32_t u = __float_as_uint(f + 0.0f);   // -0 -> +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_value(uint32_t k)
{
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

// The piece that tile `tile` of a launch belongs to (the one problem of a
// launch that is not grouped).
template <bool GROUPED>
__device__ __forceinline__ GemmPiece piece_of(int tile, const GemmPiece *pieces, int n_pieces,
                                              const GemmPiece &single)
{
    if (!GROUPED) return single;
    int lo = 0, hi = n_pieces - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pieces[mid].tile_begin <= tile) lo = mid;
        else hi = mid - 1;
    }
    return pieces[lo];
}

// The driver's tensor-map encoder, looked up once (concurrent first calls find the same one).
inline PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

inline bool get_encoder()
{
    if (g_encode) return true;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return false;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return true;
}

// 2D tensor [outer, inner] row-major (FP16, BF16 or FP8 bytes), box
// [box_outer, BK], swizzle matching the mode's row width.
template <int MODE>
bool make_map(CUtensorMap *m, const void *base, int64_t inner, int64_t outer, int box_outer)
{
    using M = Elem<MODE>;
    const int esize = MODE == kSimFp8 ? 1 : 2;
    const CUtensorMapDataType dt = MODE == kSimF16x3 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                   : (MODE == kSimBf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8);
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)inner * esize};
    cuuint32_t box[2] = {(cuuint32_t)M::BK, (cuuint32_t)box_outer};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(m, dt, 2, const_cast<void *>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE,
                          MODE == kSimF16x3 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace farm
