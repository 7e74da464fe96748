// Tensor maps of a segment's rows: X [rows][128] fp16 in boxes of 64 rows by 64 channels, 128-byte swizzle.  In shared memory a box is
// 64 rows of 128 bytes whose 16-byte pieces change places with the row: piece c of row i lies at i * 128 + ((c ^ (i & 7)) << 4),
// so that the same piece of eight rows hits different banks without padding, and one thread requests a box at once.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gear_pi.cuh"

namespace gear {

constexpr int kBoxRows = 64, kBoxChannels = 64, kBoxBytes = kBoxRows * kBoxChannels * 2;

inline cudaError_t make_row_map(CUtensorMap* map, const void* rows, long long n_rows) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                             const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess) {
      cudaGetLastError();
      fn = nullptr;
    }
    return reinterpret_cast<Encode>(fn);
  }();
  if (encode == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {kHeadDim, (cuuint64_t)n_rows}, strides[1] = {kHeadDim * 2};
  const cuuint32_t box[2] = {kBoxChannels, kBoxRows}, steps[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(rows), dims, strides, box, steps,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// box of 64 channels from channel `x` (a multiple of 64), 64 rows from `row` on; dst 1024-byte aligned
__device__ __forceinline__ void load_box(void* dst, const CUtensorMap* map, int x, int row, uint64_t* b) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_addr(dst)), "l"(map), "r"(x), "r"(row), "r"(smem_addr(b)) : "memory");
}
// byte of channel ch (below 64) of row i in a box
__device__ __forceinline__ int box_at(int i, int ch) { return i * 128 + (((ch >> 3) ^ (i & 7)) << 4) + (ch & 7) * 2; }

}  // namespace gear
