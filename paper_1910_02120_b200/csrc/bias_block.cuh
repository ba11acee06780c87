// The bias gradient and update as blocks of a launch: of bias_sgd_kernel, or behind the tiles of an fp32
// weight-update launch.
#pragma once

#include "kernels.h"

namespace ist {
namespace {

__device__ __forceinline__ void load8(const float* p, float v[8]) {
  float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const bf16* p, float v[8]) {
  uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) { v[2 * i] = __low2float(h[i]); v[2 * i + 1] = __high2float(h[i]); }
}

// Block `blk` of bias_blocks(): group blk % G, and blk / G runs over the layers' blocks of 64 columns one layer
// after the other (layer i owns xstart[i] .. xstart[i + 1] - 1).  Threads 0..255: thread (cx, ry) sums 8
// adjacent columns over rows ry, ry + 32, ...; the 32 partial sums of a column are added in a fixed
// order.  When a loss is wanted, one block more per group averages the step's row losses (fixed order).
// Called by all threads of the block.
template <typename T>
__device__ __forceinline__ void bias_block(const BiasSgdArgs<T>& a, int blk, int tid, float (*part)[65]) {
  const int g = blk % a.G, B = a.B;
  blk /= a.G;
  const bool loss = blk == a.xstart[a.n_layers];
  int li = 0;
  while (!loss && li + 1 < a.n_layers && blk >= a.xstart[li + 1]) ++li;
  const int c_blk = loss ? 0 : (blk - a.xstart[li]) * 64;
  if (tid < 256) {
    if (loss) {
      float acc = 0.f;
      for (int b = tid; b < B; b += 256) acc += a.loss.row_loss[(int64_t)g * B + b];
      for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if ((tid & 31) == 0) part[0][tid >> 5] = acc;
    } else {
      const BiasSgdLayer<T>& L = a.layer[li];
      const int cx = tid & 7, ry = tid >> 3;
      const int c0 = c_blk + cx * 8;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (c0 < L.ld) {
        const T* d = L.delta + (int64_t)g * L.sg + c0;
#pragma unroll 8
        for (int b = ry; b < B; b += 32) {
          float v[8];
          load8(d + (int64_t)b * L.ld, v);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += v[e];
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) part[ry][cx * 8 + e] = acc[e];
    }
  }
  __syncthreads();
  if (loss) {
    if (tid < 32) {
      float acc = tid < 8 ? part[0][tid] : 0.f;
      for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (tid == 0) a.loss.loss_out[(int64_t)g * a.loss.out_stride + a.loss.k] = acc / (float)B;
    }
  } else if (tid < 64) {
    const BiasSgdLayer<T>& L = a.layer[li];
    const int col = c_blk + tid;
    if (col < L.n) {
      float s = 0.f;
#pragma unroll
      for (int u = 0; u < 32; ++u) s += part[u][tid];
      L.bias[(int64_t)g * L.bias_sg + col] -= a.lr * s;
    }
  }
}

}  // namespace
}  // namespace ist
