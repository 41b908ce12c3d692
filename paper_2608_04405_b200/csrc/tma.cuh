// Key tiles by TMA: one thread brings 128 rows x 128 channels (bf16) into shared memory in the 128-byte-swizzled operand
// layout (two boxes of 64 channels), completing on an mbarrier.  Copying the tile in 16-byte pieces by all threads of a
// warpgroup cost it about 1700 cycles per tile in instruction issue and queueing next to its other work.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "umma.cuh"

namespace tma {

constexpr int kTileRows = 128;
constexpr unsigned kTileBytes = kTileRows * 256;

// Tensor map of a bf16 cache seen as `rows` rows of 128 channels, row_stride elements apart.
inline cudaError_t make_key_map(CUtensorMap* map, const void* base, unsigned long long rows, int row_stride) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                             const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = []() -> Encode {             // (looked up once; thread-safe static)
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
      (void)cudaGetLastError();
      return nullptr;
    }
    return reinterpret_cast<Encode>(fn);
  }();
  if (encode == nullptr) return cudaErrorSymbolNotFound;
  if (rows == 0 || rows > 0x7fffffffull) return cudaErrorInvalidValue;        // (row coordinates are 32-bit)
  const cuuint64_t dims[2] = {BPC_D, rows}, strides[1] = {(cuuint64_t)row_stride * 2};
  const cuuint32_t box[2] = {64, kTileRows}, step[2] = {1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, step,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

#ifdef __CUDACC__
// One thread: rows [row, row + 128) into `tile` (1024-byte aligned), arriving on `bar` when the bytes are there.  Rows past
// the map's last are zeros; rows past a unit's last key are whatever the cache holds there.
__device__ __forceinline__ void load_key_tile(unsigned char* tile, const CUtensorMap* map, int row, unsigned long long* bar) {
  const unsigned b = umma::smem_u32(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(kTileBytes) : "memory");
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(umma::smem_u32(tile + h * kTileRows * 128)), "l"(map), "r"(64 * h), "r"(row), "r"(b) : "memory");
}
#endif

}  // namespace tma
