// Host-side construction of the tensor maps that the bulk-tensor copies take.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace adaption {

// The two encoders of the driver, looked up once per process; false if either is missing.
bool load_tensor_map_encoders();

// Byte tensor of `rank` dimensions (innermost first), strides in bytes for dimensions 1.., a box per copy
// and a step per dimension (estr null: all ones).
// `long_rows`: the copies walk along rows much longer than the box, so L2 fetches 256 bytes at a time
// (a weight matrix of 4096 rows of 25088 bytes read once: 41.1 -> 36.9 us for the layer).
bool encode_tiled(CUtensorMap* map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                  const uint32_t* box, const uint32_t* estr, CUtensorMapSwizzle swz, bool long_rows = false);

// The same over elements of 8 bytes without swizzle: boxes of up to 256 of them, copied as contiguous rows.
bool encode_tiled_words(CUtensorMap* map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                        const uint32_t* box);

inline bool encode_tiled_2d(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint64_t pitch_bytes,
                            uint32_t box_inner, uint32_t box_rows, CUtensorMapSwizzle swz, bool long_rows = false) {
  const uint64_t dims[2] = {inner, rows}, strides[1] = {pitch_bytes};
  const uint32_t box[2] = {box_inner, box_rows};
  return encode_tiled(map, base, 2, dims, strides, box, nullptr, swz, long_rows);
}

// NHWC activations in im2col mode: `pixels` output pixels of one filter tap per copy.
bool encode_im2col_nhwc(CUtensorMap* map, const void* base, const adaption_conv_shape& s, int64_t c_stride,
                        uint32_t channels_per_pixel, uint32_t pixels, CUtensorMapSwizzle swz);

}  // namespace adaption
