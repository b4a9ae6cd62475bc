// Tensor maps of packed matrices, for the products that load words by TMA
// (internal).
#pragma once
#include <atomic>
#include <cuda.h>
#include "common.cuh"

namespace jsim {

namespace {

using PFN_encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                               const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder (null: not available).
inline PFN_encode tensor_map_encoder()
{
    static std::atomic<void*> fn{nullptr};
    void* p = fn.load(std::memory_order_acquire);
    if (!p) {
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        fn.store(p, std::memory_order_release);
    }
    return (PFN_encode)p;
}

// The tensor map of a packed matrix (n rows of W words, `stride` apart) in
// boxes of 128 rows x `box_words` words; false where the rows are not 16-byte
// aligned (or the encoder refuses).
inline bool packed_map(CUtensorMap* map, const u64* X, u64 n, u64 W, u64 stride, u32 box_words, CUtensorMapSwizzle swz)
{
    if ((uintptr_t)X % 16 != 0 || stride % 2 != 0 || W == 0 || n == 0 || W >= (1ull << 31) || stride * 8 >= (1ull << 40))
        return false;
    PFN_encode enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {W, n}, strides[1] = {stride * 8};
    const cuuint32_t box[2] = {box_words, 128}, estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, (void*)X, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

}  // namespace jsim
