// Shared definitions of the IST library's device code: status word, launch helpers, types.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ist {

typedef __nv_bfloat16 bf16;

// Sticky device status: word 0 = code (0 = ok, otherwise an ist_status value), word 1 = site
// tag of the first failure, words 2..3 = detail (offending index / value).
struct DeviceStatus {
  int code;
  int site;
  long long detail;
};

enum Site : int {
  SITE_NONE = 0,
  SITE_LABEL = 1,      // label outside [0, N_t)
  SITE_CSR_COL = 2,    // CSR column outside [0, N_0)
  SITE_PART_IDX = 3,   // partition index outside [0, N_l)
  SITE_TC_PIPE = 4,    // bounded wait in the tensor-core pipeline expired
  SITE_CSR_ROW = 5     // CSR row_ptr not monotone
};

__device__ __forceinline__ void report(DeviceStatus* st, int code, int site, long long detail) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->site = site;
    st->detail = detail;
  }
}

// Programmatic dependent launch.  A kernel launched with launch_pdl may be scheduled while the
// kernel before it in the stream is still running; it must call pdl_wait() before it touches
// global memory (that waits until the earlier kernel has completed and its writes are visible).
// pdl_trigger() lets the kernel after this one be scheduled as this grid's CTAs retire.
// Such a kernel reads with plain loads only, no __ldg and no `const __restrict__` parameters: the
// non-coherent path asks for data that is constant for the kernel's whole life, which begins while the
// earlier kernel may still be writing it, and the compiler may move those loads ahead of the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

__host__ __device__ __forceinline__ constexpr int64_t ceil_div(int64_t a, int64_t b) {
  return (a + b - 1) / b;
}
__host__ __device__ __forceinline__ constexpr int64_t round_up(int64_t a, int64_t b) {
  return ceil_div(a, b) * b;
}

// An fp32 master and the bf16 operand made from it take 32 bits together: the operand is the master rounded to
// its upper 16 bits, ties away from zero, and beside it lie the lower 16 bits of the master; the operand's last bit and
// the low half's first say whether the rounding went up, so the master comes back bit for bit.  (With ties to
// even, two masters would share an operand and a low half.)  A weight update then moves 8 bytes per weight
// instead of 10.  NaNs become one NaN: their payloads do not fit.
__device__ __forceinline__ void split_master(float w, uint16_t* hi, uint16_t* lo) {
  uint32_t u = __float_as_uint(w);
  if (w != w) u = 0x7fc00000u;
  *hi = (uint16_t)((u + 0x8000u) >> 16);
  *lo = (uint16_t)u;
}
__device__ __forceinline__ float join_master(uint16_t hi, uint16_t lo) {
  return __uint_as_float(((uint32_t)hi << 16) + (uint32_t)(int)(int16_t)lo);
}
__device__ __forceinline__ uint16_t operand_bits(float w) {
  uint16_t hi, lo;
  split_master(w, &hi, &lo);
  return hi;
}

// Bits of an updated master.  The NaN that arithmetic gives, 0x7fffffff, would round to minus zero: the signed minimum
// makes it one that stays a NaN and leaves every number as it is.
__device__ __forceinline__ uint32_t master_bits(float w) { return (uint32_t)min(__float_as_int(w), 0x7fff7fff); }
// The operands of eight masters (see split_master), as one 16-byte unit.
__device__ __forceinline__ uint4 pack8_operand(const float* w) {
  uint32_t h[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) h[e] = master_bits(w[e]) + 0x8000u;
  return make_uint4(__byte_perm(h[0], h[1], 0x7632), __byte_perm(h[2], h[3], 0x7632), __byte_perm(h[4], h[5], 0x7632),
                    __byte_perm(h[6], h[7], 0x7632));
}
// Eight masters kept as operand and low half: joined, and taken apart again.
__device__ __forceinline__ void join8(const uint4& h, const uint4& l, float* w) {
  const uint32_t hv[4] = {h.x, h.y, h.z, h.w}, lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    w[2 * i] = __uint_as_float((hv[i] << 16) + (uint32_t)((int)(lv[i] << 16) >> 16));
    w[2 * i + 1] = __uint_as_float((hv[i] & 0xffff0000u) + (uint32_t)((int)lv[i] >> 16));
  }
}
__device__ __forceinline__ void split8(const float* w, uint4* h, uint4* l) {
  uint32_t v[8], hv[4], lv[4];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = master_bits(w[e]);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    hv[i] = __byte_perm(v[2 * i] + 0x8000u, v[2 * i + 1] + 0x8000u, 0x7632);
    lv[i] = __byte_perm(v[2 * i], v[2 * i + 1], 0x5410);
  }
  *h = make_uint4(hv[0], hv[1], hv[2], hv[3]);
  *l = make_uint4(lv[0], lv[1], lv[2], lv[3]);
}

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_float(float v);
template <> __device__ __forceinline__ float from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_float<bf16>(float v) { return __float2bfloat16_rn(v); }

// Four adjacent elements as one 16-byte (fp32) or 8-byte (bf16) access; p must be aligned to it.
__device__ __forceinline__ void load4(const float* p, float v[4]) {
  float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const bf16* p, float v[4]) {
  uint2 t = *reinterpret_cast<const uint2*>(p);
  __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&t.x);
  __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162*>(&t.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}
__device__ __forceinline__ void store4(float* p, const float v[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(bf16* p, const float v[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
  __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
  uint2 t;
  t.x = *reinterpret_cast<uint32_t*>(&a);
  t.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = t;
}

}  // namespace ist
