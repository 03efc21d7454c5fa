#include "tensor_maps.cuh"

#include <mutex>

namespace adaption {
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn g_encode_tiled = nullptr;
EncodeIm2colFn g_encode_im2col = nullptr;
std::once_flag g_encode_once;

}  // namespace

// (they are the same for every device)
bool load_tensor_map_encoders() {
  std::call_once(g_encode_once, [] {
    void* f1 = nullptr;
    void* f2 = nullptr;
    cudaDriverEntryPointQueryResult q1, q2;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f1, cudaEnableDefault, &q1) != cudaSuccess ||
        q1 != cudaDriverEntryPointSuccess || f1 == nullptr)
      return;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &f2, cudaEnableDefault, &q2) != cudaSuccess ||
        q2 != cudaDriverEntryPointSuccess || f2 == nullptr)
      return;
    g_encode_im2col = reinterpret_cast<EncodeIm2colFn>(f2);
    g_encode_tiled = reinterpret_cast<EncodeTiledFn>(f1);
  });
  return g_encode_tiled != nullptr && g_encode_im2col != nullptr;
}

static bool encode(CUtensorMap* map, CUtensorMapDataType type, const void* base, int rank, const uint64_t* dims,
                   const uint64_t* strides, const uint32_t* box, const uint32_t* estr, CUtensorMapSwizzle swz, bool long_rows) {
  cuuint64_t d[5], s[4];
  cuuint32_t b[5], e[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    e[i] = estr != nullptr ? estr[i] : 1u;
    if (i > 0) s[i - 1] = strides[i - 1];
  }
  return g_encode_tiled(map, type, (cuuint32_t)rank, const_cast<void*>(base), d, s, b, e,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                        long_rows ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_tiled(CUtensorMap* map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                  const uint32_t* box, const uint32_t* estr, CUtensorMapSwizzle swz, bool long_rows) {
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, base, rank, dims, strides, box, estr, swz, long_rows);
}

bool encode_tiled_words(CUtensorMap* map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                        const uint32_t* box) {
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_INT64, base, rank, dims, strides, box, nullptr, CU_TENSOR_MAP_SWIZZLE_NONE, false);
}

bool encode_im2col_nhwc(CUtensorMap* map, const void* base, const adaption_conv_shape& s, int64_t c_stride,
                        uint32_t channels_per_pixel, uint32_t pixels, CUtensorMapSwizzle swz) {
  cuuint64_t dims[4] = {(cuuint64_t)c_stride, (cuuint64_t)s.W, (cuuint64_t)s.H, (cuuint64_t)s.N};
  cuuint64_t strides[3] = {(cuuint64_t)c_stride, (cuuint64_t)c_stride * s.W,
                           (cuuint64_t)c_stride * s.W * s.H};
  int lower[2] = {-s.pad_w, -s.pad_h};
  int upper[2] = {s.pad_w - (s.S - 1), s.pad_h - (s.R - 1)};
  cuuint32_t estr[4] = {1, (cuuint32_t)s.stride_w, (cuuint32_t)s.stride_h, 1};
  return g_encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base), dims, strides,
                         lower, upper, channels_per_pixel, (cuuint32_t)pixels, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace adaption
