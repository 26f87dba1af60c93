// Tensor maps for tiled bulk copies (TMA), encoded by the driver and kept.
#pragma once

#include <cuda.h>

namespace seqtree {

// Encodes a map with 128-byte swizzle and zero fill; strides in bytes, for dimensions 1 .. rank-1.  False if the driver
// refuses.
bool tensor_map(CUtensorMap* out, CUtensorMapDataType type, unsigned rank, const void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t* box);

}  // namespace seqtree
