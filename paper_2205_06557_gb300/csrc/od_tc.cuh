// Fifth-generation tensor cores and the tensor memory accelerator, as the network's kernels
// use them (od_gemm_tc.cu, od_mlp.cu): shared-memory and instruction descriptors, mbarriers with
// bounded waits, tensor-memory reads, tensor maps.
#pragma once

#include <cuda.h>  // CUtensorMap and the encoder's types; the encoder itself is fetched
                   // through the runtime's entry-point query (no link to libcuda)
#include <cuda_bf16.h>

#include <cstdint>
#include <mutex>

#include "od_internal.h"

namespace od {
namespace tc {

constexpr long long WAIT_LIMIT = 1ll << 22;  // polls of an mbarrier before giving up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor of a K-major tile in the 128-byte swizzled layout:
// start address, leading byte offset 16 (unused for this layout), stride byte offset
// 1,024 (8 rows of 128 bytes), descriptor version 1, layout type 2 (SWIZZLE_128B)
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major
__device__ __forceinline__ uint32_t instr_desc(int m, int n)
{
    return (1u << 4)                        // D format: F32
           | (1u << 7)                      // A format: BF16
           | (1u << 10)                     // B format: BF16
           | ((uint32_t)(n >> 3) << 17)     // N / 8
           | ((uint32_t)(m >> 4) << 24);    // M / 16
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait for the phase with this parity to complete; false if it did not
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity)
{
    for (long long it = 0; it < WAIT_LIMIT; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// tcgen05.ld of W = 16 or 32 consecutive accumulator columns of the warp's 32 lanes (rows),
// issued without waiting; tmem_wait(v) waits for every load the thread issued and names v as
// its operands, so that no use of v moves before it
template <int W>
__device__ __forceinline__ void tmem_issue(uint32_t taddr, uint32_t (&v)[W]);

template <>
__device__ __forceinline__ void tmem_issue<16>(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}

template <>
__device__ __forceinline__ void tmem_issue<32>(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
}

template <int W>
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[W])
{
#pragma unroll
    for (int e = 0; e < W; e += 16)
        asm volatile("" : "+r"(v[e]), "+r"(v[e + 1]), "+r"(v[e + 2]), "+r"(v[e + 3]), "+r"(v[e + 4]), "+r"(v[e + 5]),
                     "+r"(v[e + 6]), "+r"(v[e + 7]), "+r"(v[e + 8]), "+r"(v[e + 9]), "+r"(v[e + 10]), "+r"(v[e + 11]),
                     "+r"(v[e + 12]), "+r"(v[e + 13]), "+r"(v[e + 14]), "+r"(v[e + 15])::"memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < W; e += 16)
        asm volatile("" : "+r"(v[e]), "+r"(v[e + 1]), "+r"(v[e + 2]), "+r"(v[e + 3]), "+r"(v[e + 4]), "+r"(v[e + 5]),
                     "+r"(v[e + 6]), "+r"(v[e + 7]), "+r"(v[e + 8]), "+r"(v[e + 9]), "+r"(v[e + 10]), "+r"(v[e + 11]),
                     "+r"(v[e + 12]), "+r"(v[e + 13]), "+r"(v[e + 14]), "+r"(v[e + 15])::"memory");
}

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiled encoder()
{
    static EncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiled)p;
        cudaGetLastError();
    });
    return fn;
}

// a rows x K BF16 row-major matrix, read in boxes of box_rows x 64 with the 128-byte swizzle;
// reads past the matrix return zeros
inline bool encode_tiled(CUtensorMap* tm, const __nv_bfloat16* base, int rows, int K, int box_rows)
{
    const EncodeTiled fn = encoder();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


}  // namespace tc
}  // namespace od
