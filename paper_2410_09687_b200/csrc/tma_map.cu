// Tensor maps and shape predicates of the tcgen05 kernels.
#include <cuda.h>

#include "tc_gemm.cuh"

namespace moin {

constexpr int kMapBox = 64;   // elements of a box row: 128 bytes, one swizzle row

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

static moin_status get_encoder() {
  if (g_encode) return MOIN_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess) return record_cuda(e);
  if (qres != cudaDriverEntryPointSuccess || !fn) return record_cuda(cudaErrorNotSupported);
  g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  return MOIN_OK;
}

// 2-D row-major bf16 tensor [rows, cols] -> map with a [box_rows x 64] box, 128-byte swizzle, zero fill.
moin_status make_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  moin_status st = get_encoder();
  if (st) return st;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kMapBox, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return record_cuda(cudaErrorInvalidValue);
  return MOIN_OK;
}

// 2-D row-major byte tensor [rows, cols] -> map with a [box_rows x 64] box, 64-byte swizzle, zero fill.
moin_status make_map_u8(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  moin_status st = get_encoder();
  if (st) return st;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols};
  cuuint32_t box[2] = {(cuuint32_t)kMapBox, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return record_cuda(cudaErrorInvalidValue);
  return MOIN_OK;
}

// bf16 [T][n_heads][64] -> map with a box of box_t tokens x box_heads heads x 64, 128-byte swizzle, zero fill.
moin_status make_map_heads(CUtensorMap* map, const void* base, uint64_t T, uint32_t n_heads, uint32_t box_heads, uint32_t box_t) {
  moin_status st = get_encoder();
  if (st) return st;
  cuuint64_t dims[3] = {(cuuint64_t)kMapBox, n_heads, T};
  cuuint64_t strides[2] = {kMapBox * 2, (cuuint64_t)n_heads * kMapBox * 2};
  cuuint32_t box[3] = {(cuuint32_t)kMapBox, box_heads, box_t};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return record_cuda(cudaErrorInvalidValue);
  return MOIN_OK;
}

bool tc_gemm_supported(int T, int d_in, int d_out) { return T >= 1 && d_in >= 64 && (d_in % 8) == 0 && (d_out % 8) == 0; }
bool tc_router_supported(int Q, int K, int D) { return Q >= 1 && K >= 1 && D >= 64 && (D % 8) == 0; }
bool tc_fused_supported(int r) { return r >= 8 && r <= 128 && (r % 8) == 0; }

}  // namespace moin
