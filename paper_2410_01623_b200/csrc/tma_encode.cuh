// Tensor-map encoding on the host.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace fira {

// A bf16 or fp32 tensor of `rank` (2 to 4) dimensions, innermost first: extents, byte strides of the outer
// dimensions and box.  swizzle_bytes: 128, 64 or 0.  Elements outside the extents load as zeros.
bool encode_tiled(CUtensorMap* out, const void* base, bool fp32, int rank, const unsigned long long* extent,
                  const unsigned long long* stride_bytes, const unsigned* box, int swizzle_bytes);

}  // namespace fira
