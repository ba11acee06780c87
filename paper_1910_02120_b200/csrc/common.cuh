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

// An fp32 master and the bf16 operand made from it take 32 bits together: the operand is the master rounded to its
// upper 16 bits (to nearest, ties to even), and beside it lie the lower 16 bits of the master; the operand's last bit
// and the low half's first say whether the rounding went up, so the master comes back.  A weight update then moves 8
// bytes per weight instead of 10.  Only the two ties that round to the same even operand look alike: a bit per master, a
// sixty-fourth of the traffic, is set for the one that rounded down, and counts only where operand and low half are such a
// pair's.  Every number comes back bit for bit, and a NaN as a NaN.  (Rounding ties away from zero would need no bit, but
// changes the operand of one weight in 2^17 by 2^-8, which turns ReLU masks over.)
__device__ __forceinline__ float join_master(uint16_t hi, uint16_t lo) {   // of two ties, the one that rounded up
  return __uint_as_float(((uint32_t)hi << 16) + (uint32_t)(int)(int16_t)lo);
}
__device__ __forceinline__ bool may_be_tie(float joined) { return (__float_as_uint(joined) & 0x1ffffu) == 0x18000u; }
__device__ __forceinline__ float other_tie(float joined) { return __uint_as_float(__float_as_uint(joined) + 0x10000u); }
// Tie bits: words of 32 columns, [slab][columns / 32][rows], so that a warp on consecutive rows reads consecutive words.
// Column 2 i of the 32 has bit 15 - i, column 2 i + 1 bit 31 - i (see split8).
__host__ __device__ __forceinline__ constexpr int64_t tie_words(int64_t rows, int64_t ld) { return (ld + 31) / 32 * rows; }   // of a slab
struct TieBit {
  int64_t word;
  uint32_t mask;
};
__device__ __forceinline__ TieBit tie_bit(int64_t rows, int64_t ld, int64_t slab, int64_t row, int64_t col) {
  return TieBit{slab * tie_words(rows, ld) + (col >> 5) * rows + row, 1u << (15 - ((int)col & 31) / 2 + ((int)col & 1) * 16)};
}

// Eight masters kept as operand and low half: joined, and taken apart again.
__device__ __forceinline__ void join8(const uint4& h, const uint4& l, float* w) {
  const uint32_t hv[4] = {h.x, h.y, h.z, h.w}, lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t b = lv[i] ^ 0x80008000u;                  // the low half plus 2^15: no sign to extend
    w[2 * i] = __uint_as_float(__byte_perm(b, hv[i], 0x5410) - 0x8000u);
    w[2 * i + 1] = __uint_as_float(__byte_perm(b, hv[i], 0x7632) - 0x8000u);
  }
}
// Operands and low halves of two masters.  Ties that rounded down are where adding half an operand's ulp and cutting gives the
// odd neighbour of the operand: bit 0 or 16 of *ties.
__device__ __forceinline__ void split2(float w0, float w1, uint32_t* h, uint32_t* l, uint32_t* ties) {
  const uint32_t u0 = __float_as_uint(w0), u1 = __float_as_uint(w1);
  const __nv_bfloat162 o = __floats2bfloat162_rn(w0, w1);
  *h = *reinterpret_cast<const uint32_t*>(&o);
  *l = __byte_perm(u0, u1, 0x5410);
  *ties = (__byte_perm(u0 + 0x8000u, u1 + 0x8000u, 0x7632) ^ *h) & 0x00010001u;
}
// The tie bits are shifted in, two a step: sixteen steps make a word.
__device__ __forceinline__ void split8(const float* w, uint4* h, uint4* l, uint32_t* ties) {
  uint32_t hv[4], lv[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t t;
    split2(w[2 * i], w[2 * i + 1], &hv[i], &lv[i], &t);
    *ties = *ties * 2u + t;
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
