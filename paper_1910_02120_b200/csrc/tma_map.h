// Host side of the tensor maps that the tensor-core kernels copy through (defined in gemm_tc.cu).
#pragma once

#include <cuda.h>

namespace ist {

int sm_count();
// Tensor [groups][outer][inner] (inner contiguous, strides in elements) with box
// {box_inner, box_outer, 1}.  elem_bytes 2 = 16-bit values, 4 = fp32.  swizzle_bytes 128 or 64.
bool make_map(CUtensorMap* out, const void* base, int elem_bytes, long long inner, long long outer, long long groups,
              long long outer_stride, long long group_stride, int box_inner, int box_outer, int swizzle_bytes);

}  // namespace ist
