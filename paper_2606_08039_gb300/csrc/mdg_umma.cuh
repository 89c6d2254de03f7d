// Shared by the tcgen05 kernels of the surrogate network (inference in mdg_umma.cu, training in
// mdg_train.cu): the 128-byte-swizzled operand layout and its descriptors, the weight image,
// bounded mbarrier waits, tensor-memory loads and the TMA of an input tile.
#ifndef MDG_UMMA_CUH
#define MDG_UMMA_CUH

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "mdg.h"
#include "mdg_internal.cuh"

namespace mdg {
namespace {

constexpr int kRows = 128;                 // tile rows (UMMA M)
constexpr int kEpiWarps = 16;              // four per TMEM lane quadrant
constexpr uint32_t kSlotBytes = 32768;     // one [256 x 64] bf16 weight chunk
constexpr uint32_t kChunkBytes = 16384;    // one [128 x 64] bf16 activation chunk
constexpr uint32_t kTmemCols = 512;        // two accumulators of 256 columns
constexpr uint32_t kSuspendNs = 1000;      // longest suspension of one mbarrier try_wait
constexpr int kWaitLimit = MDG_MLP_DEFAULT_TRY_WAITS;  // try_waits (at most ~0.26 s) before giving up

// Weight image: the chunks in the order the MMAs consume them, load i at i * 32 KB.
//   load 0      W1 [256 x 64]
//   loads 1-4   W2 chunk c [256 x 64]
//   loads 5-8   W3 chunk c [256 x 64]
//   load 9      W4 [32 x 256] as four [32 x 64] chunks of 4 KB (16 KB)
constexpr uint32_t kImgBytes = 9 * kSlotBytes + 16384;
static_assert(kImgBytes == 2 * (256 * 64 + 2 * 256 * 256 + 32 * 256), "the image holds every weight once");

__device__ __forceinline__ uint32_t image_layer_base(int l)
{
    return l == 0 ? 0u : l == 1 ? kSlotBytes : l == 2 ? 5 * kSlotBytes : 9 * kSlotBytes;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);  // start address
    d |= (uint64_t)1 << 16;                           // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                           // descriptor version
    d |= (uint64_t)2 << 61;                           // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 A and B (K-major), FP32 D, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16_ss(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// The mbarrier completes once every tcgen05 operation issued so far by this thread is done.
__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    return done != 0;
}

// Wait for the phase of `parity` to complete: one non-blocking test, then mbarrier.try_wait,
// which suspends the thread in hardware until the phase completes or about kSuspendNs pass.
// Gives up when another role has aborted (abort != null) or after `limit` tries, which
// records the timeout and aborts the block. The work waits take the launch's limit; the
// drain waits of the exit path always take kWaitLimit, so that a block leaves only once
// every copy and MMA it issued has completed.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, volatile int* abort, uint32_t* status,
                                          int limit)
{
    if (mbar_test(mbar, parity)) return true;
    for (int i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity), "r"(kSuspendNs)
            : "memory");
        if (done) return true;
        if (abort && *abort) return false;
    }
    if (abort) *abort = 1;
    atomicOr(status, MDG_STATUS_TIMEOUT);
    return false;
}

// The same for waits on the critical path between MMAs and epilogue: poll with test_wait
// (a suspended thread wakes up later than a polling one), backing off by `sleep_ns` between
// polls (0: none), at most `limit` polls.
__device__ __forceinline__ bool mbar_spin(uint32_t mbar, uint32_t parity, volatile int* abort, uint32_t* status,
                                          int sleep_ns, int limit)
{
    for (int i = 0; i < limit; ++i) {
        if (mbar_test(mbar, parity)) return true;
        if ((i & 63) == 63 && *abort) return false;
        if (sleep_ns) __nanosleep(sleep_ns);
    }
    *abort = 1;
    atomicOr(status, MDG_STATUS_TIMEOUT);
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
}

// Bulk copy global -> shared; completes `bytes` of the mbarrier's transaction count.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t s, const void* g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(g));
}

// 16 (x16) or 8 (x8) consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float v[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// TMA of one [128 x 64] bf16 input tile (rows row..row+127) into 128-byte-swizzled shared
// memory, completing on mbar; and its prefetch into L2.
__device__ __forceinline__ void tma_rows(uint32_t dst, const CUtensorMap* map, int row, uint32_t mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(mbar) : "memory");
}
__device__ __forceinline__ void tma_rows_prefetch(const CUtensorMap* map, int row)
{
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];\n"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row) : "memory");
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// cuTensorMapEncodeTiled, looked up through the runtime (no link against the driver library).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiledFn encode_tiled()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// The tensor map of the network inputs x [B x 64] bf16, row-major: boxes of one tile (128 rows
// x 128 bytes), 128-byte swizzle. x must be 16-byte aligned.
inline cudaError_t input_map(CUtensorMap* map, const void* x, int B)
{
    if (reinterpret_cast<uintptr_t>(x) % 16) return cudaErrorMisalignedAddress;  // TMA source
    const EncodeTiledFn encode = encode_tiled();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {MDG_MLP_IN_PAD, (cuuint64_t)B};
    const cuuint64_t strides[1] = {MDG_MLP_IN_PAD * sizeof(__nv_bfloat16)};
    const cuuint32_t box[2] = {MDG_MLP_IN_PAD, kRows};
    const cuuint32_t elem_strides[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), dims, strides, box, elem_strides,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}


}  // namespace
}  // namespace mdg

#endif  // MDG_UMMA_CUH
