// TMA tensor maps, encoded through the runtime's driver entry point.
#pragma once

#include <cuda.h>
#include <cstdint>

namespace last {

// A bf16 tensor of `rank` dimensions (inner first; `strides` in bytes, of dimensions 1
// up) with the 128-byte swizzle and zero fill; the box's inner extent is 64 elements.
bool encode_bf16_map(CUtensorMap *m, const void *base, int rank, const uint64_t *dims,
                     const uint64_t *strides, const uint32_t *box);

}  // namespace last
