// Whole tiles of the temporal form's activations and gradients by TMA, shared by
// the BF16 (train_tct.cu) and FP32 (train_temporal.cu) training kernels.
#pragma once
#include "et_internal.cuh"
#include "tc_ptx.cuh"
#include <cuda.h>

namespace {

// Tensors are [B K][hw][16] FP32.  A box is one step of 128 pixels: 128 rows of
// 64 bytes, 64-byte swizzled in shared memory, so that the 8 lanes of a 16-byte
// access phase, each reading its own pixel's row, meet 32 different banks
// (thread-per-pixel reads of global rows cost 16 lines per 512 bytes and left
// the kernels at 28 % of the HBM rate).  Rows beyond hw are zero-filled on loads
// and dropped on stores by the tensor map.
constexpr int kBoxPix = 128;
constexpr int kBox = kBoxPix * 16 * 4;       // bytes of one step's tile

__device__ __forceinline__ const float4* box_row(const unsigned char* box, int p, int j) {
  return reinterpret_cast<const float4*>(box + p * 64 + 16 * (j ^ ((p >> 1) & 3)));
}
__device__ __forceinline__ void box_load(const unsigned char* box, int p, float (&v)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 x = *box_row(box, p, j);
    v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
  }
}
__device__ __forceinline__ void box_store(unsigned char* box, int p, const float (&v)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<float4*>(box + p * 64 + 16 * (j ^ ((p >> 1) & 3))) =
        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}
// shared memory -> the tensor's box at (x, y, z); completes with the issuing
// thread's bulk group
__device__ __forceinline__ void tma_store_3d(const void* tmap, int x, int y, int z, const void* src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every committed store has read its shared memory / has completed
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// tensor map of [steps][hw][16] floats, box = one step of 128 pixels
inline int map_rows(CUtensorMap* m, const float* base, int64_t steps, int64_t hw) {
  typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                               const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const EncodeFn encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &qr) !=
            cudaSuccess || qr != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeFn>(f);
  }();
  if (!encode) return ET_ERR_CUDA;
  const cuuint64_t dims[3] = {16, (cuuint64_t)hw, (cuuint64_t)steps};
  const cuuint64_t strides[2] = {16 * 4, (cuuint64_t)hw * 16 * 4};
  const cuuint32_t box[3] = {16, (cuuint32_t)kBoxPix, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? ET_OK : ET_ERR_CUDA;
}

// the TMA forms: 16 channels, 16-byte aligned tensors, coordinates within 31 bits
inline bool use_tma(int B, int K, int64_t hw, int C, const float* a, const float* b) {
  return C == 16 && (int64_t)B * K < (1ll << 31) && hw < (1ll << 31) - kBoxPix &&
         ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}

}  // namespace
