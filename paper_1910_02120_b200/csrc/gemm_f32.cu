// Grouped fp32 GEMM on the 5th-generation tensor cores: the fp32 path of the local steps (forward,
// backward and SGD update of all S subnets; paper Sec. 2.1 "Training Subnets", App. A Eq. (2) on
// the slices), their input gradients, and the full-width evaluation pass.
//
//   C[g](m, n) = sum_k A[g](m, k) * B[g](n, k)
//
// Every fp32 operand is split into three bf16 numbers (8 + 8 + 8 significant bits):
// x = h + 2^-8 m + 2^-16 l with h = bf16(x), m = bf16(2^8 (x - h)), l = 2^8 (2^8 (x - h) - m).  A
// product of two of them is then nine bf16 products, of which the six of weight 2^-16 and above are formed:
//   a b = ah bh + 2^-8 (ah bm + am bh) + 2^-16 (ah bl + am bm + al bh) + O(2^-26 |a b|),
// and the three left out are below the rounding of a single fp32 multiplication (2^-24).  The weights
// are applied to the accumulator between the groups, by the MMA's own scaling of it.  The split is exact for
// every normal number: l's last bit, 2^-149 for the smallest of them, is 2^-133 in l, bf16's smallest subnormal
// number.  (With parts of their own size bits were lost from 2^-110 down: a 100-term sum of products of 2^-126 and 2^126
// was off by up to 3.9e-4, now by 1.0e-7 as at any other magnitude.  The scaling costs single-CTA products 2 to 5 %,
// pairs nothing.)
// The tensor core's own accumulation is not relied on over long sums: 32 values of k are
// accumulated in tensor memory (the small products first, so that only the last two
// instructions act on a sum of full size), and the 32-deep sums are then added up in fp32
// registers with round-to-nearest.
//
// A CTA computes a 128 x BN tile (PAIR = 2: two CTAs of a cluster a 256 x BN one, each with its own
// 128 rows of A and half of B) in steps of 32 k values.
//   warps 0..7   load fp32 operands with plain vector loads (any base, any stride: rows of the full
//                network need not be 16-byte aligned), one or two steps ahead of their use, and
//                split them into the three bf16 planes in shared memory (128-byte swizzle, two
//                slots of 32 k values; four in a pair)
//   warps 8..15  move finished 32-deep sums from tensor memory into registers, adding up
//   one thread   issues the MMAs.  It is held up for as long as they take to start (60 cycles each,
//                128 on a 256-column tile), so on narrow tiles, where adding up is quick, it has a
//                warp of its own; on 256-column tiles, where such a warp would cost the
//                other sixteen a quarter of their registers, it sits in warp 8
// Three barriers per slot / accumulator connect them:
//   full[s]   every loading warp has written its part of slot s
//   done[s]   the MMAs on slot s are complete: their accumulator can be read, slot s rewritten
//   taken[b]  every adding warp has read accumulator b: the MMAs after next may overwrite it
// In a pair the MMAs of one CTA read both CTAs' slots.  That the other CTA's slot is written is passed on by one
// thread on either side (peer[s]): it waits for its own CTA's loading warps, releases at cluster scope, and
// is acquired there at cluster scope before it counts towards full[s].  Done two steps ahead by an
// adding warp, the release (most of a microsecond) is off the chain; with a release by every loading
// warp instead, which also waits for its loads in flight, 512 x 16384 x 16384 takes 1.3 times as long.
// Against arrivals of the loading warps without cluster scope, which nothing orders against the MMAs' reads,
// it costs 3 %.  taken[b] carries no memory, only completed tensor-memory reads, and is a relaxed
// arrival at cluster scope.
//
// A product with few tiles is cut along k over the CTAs of a cluster (up to eight); each leaves
// its sums in shared memory and the cluster adds them up in rank order, every CTA finishing its
// share of the tile's rows.
//
// Values that have no such decomposition (infinities, NaN, and magnitudes that round to infinity
// in bf16) turn the products they enter into NaN.  Every result that is not finite is computed again
// as a chain of fp32 multiply-adds, see redo(), so that the outcome is the one of fp32 arithmetic.
//
// What bounds it: pairs, the tensor pipe (12 MMAs per step and 256 x 256 tile, about 1540 cycles) at the
// clock the power limit leaves: 512 x 16384 x 16384 in 1.23 ms = 223 TFLOP/s of fp32 products,
// 1.34 PFLOP/s of bf16 ones (the same product on the CUDA cores, 128 x 128 tiles: 6.5 ms).  Single
// CTAs, the chain wait - split - barrier - MMA of a step, about 0.95 us (256 x 1024 x 1024 of
// four groups 164 -> 28 us, 1024 x 1024 x 256 of four groups 96 -> 25 us).  Error of a K-term sum
// against 64 bits, relative 2-norm, before -> now: K = 64 1.0e-7 -> 6e-8, 1024 4.1e-7 -> 1.2e-7,
// 16384 1.6e-6 -> 4.1e-7.  The tensor core cuts its sums off instead of rounding them: sums of
// terms of one sign come out 4.5e-8 too small on average, at any depth (terms of both signs: below 2e-8).
//
// Every wait is bounded, see tc_ptx.cuh.
#include <algorithm>
#include <cfloat>
#include <mutex>

#include "bias_block.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace ist {
namespace {

constexpr int BM = 128;
constexpr int KH = 32;                  // k values of a step
constexpr int kLoadWarps = 8, kAddWarps = 8, kThreads = 32 * (kLoadWarps + kAddWarps);   // those of finish()
// narrow tiles: a warp of its own issues the MMAs (with the three beside it that fill up its
// register-allotment group)
constexpr int threads_of(int bn) { return bn == 256 ? kThreads : kThreads + 128; }
constexpr int kMaxProblems = gemm_f32_max_batch();

struct F32Problem {
  int M, N, K, G;
  int m_tiles, n_tiles, tile_end;       // tiles tile_end(previous) .. tile_end - 1 of the launch
  int epi, vec;                         // vec bits: 1 A, 2 B loads, 4 output accesses may be 16-byte vectors
  const float* A; long long a_st, a_sg; // row stride (K-major) or k stride (MN-major), group stride
  const float* B; long long b_st, b_sg;
  const float* bias; long long bias_sg;
  float* out; long long out_ld, out_sg;
  const float* mask; long long mask_ld, mask_sg;
};

struct F32Args {
  int n_problems;
  int ksplit;                           // CTAs of a cluster that share a tile's k range
  float lr;
  DeviceStatus* status;
  F32Problem p[kMaxProblems];
  int side_ctas, side_blocks;           // CTAs behind those of the tiles, and blocks of bias work they share
  BiasSgdArgs<float> bias;
};

__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
  return v;
}
// (x, y) - (the two bf16 numbers in `part`), times 2^8: both steps are exact.  PACKED: as two-float
// instructions, which is what the loading warps of a pair, bound by issue slots, are better off with (512 x 16384 x
// 16384 1.30 against 1.33 ms); on single CTAs, bound by the chain of a step, they are in the way (300 rows of an
// evaluation of 1024-4096-4096-35 272 against 255 us).
template <bool PACKED>
__device__ __forceinline__ void rest2(float& x, float& y, uint32_t part) {
  if (PACKED) {
    uint64_t v = pack2(__float_as_uint(x), __float_as_uint(y));
    const uint64_t p = pack2(part << 16, part & 0xffff0000u), c = pack2(0x43800000u, 0x43800000u);   // 256
    uint32_t lo, hi;
    asm("sub.rn.f32x2 %0, %0, %1;" : "+l"(v) : "l"(p));
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(v) : "l"(c));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
    x = __uint_as_float(lo);
    y = __uint_as_float(hi);
  } else {
    x = (x - __uint_as_float(part << 16)) * 256.f;
    y = (y - __uint_as_float(part & 0xffff0000u)) * 256.f;
  }
}
// Two floats into their three bf16 parts, packed pairwise.
template <bool PACKED>
__device__ __forceinline__ void split2(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = cvt_bf16x2(x, y);
  rest2<PACKED>(x, y, h);
  m = cvt_bf16x2(x, y);
  rest2<PACKED>(x, y, m);
  l = cvt_bf16x2(x, y);
}
__device__ __forceinline__ void add2(uint64_t& acc, uint32_t lo, uint32_t hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(v));
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// One operand's share of a loading thread: UNITS groups of eight consecutive floats of a step.
//   K-major (rows contiguous along k): a warp takes 8 rows x 32 k, lane -> row (l / 4) % 2 * 4 + l / 8,
//     eight k from l % 4 * 8, unit i 64 rows further; the two rows of eight lanes differ by 4, so that
//     their swizzled 16-byte stores meet eight different bank groups.
//   MN-major (contiguous along m or n): a warp takes 4 k x 64 columns, unit i 64 columns further.
template <int MN, int UNITS>
struct Operand {
  const float* p;
  long long unit_step, half_step;
  int rows;          // K-major: rows left from this thread's first one; MN-major: columns left
  int kofs;          // first k of this thread inside a step
  uint32_t off0;     // offset inside the operand's plane, slot 0
  bool vec;
  __device__ __forceinline__ void init(const float* base, long long st, int row0, int extent, int k0, int tid, bool v) {
    const int warp = tid >> 5, lane = tid & 31;
    vec = v;
    if (MN) {
      const int k = warp * 4 + (lane >> 3), col = (lane & 7) * 8;
      kofs = k;
      p = base + (long long)(k0 + k) * st + row0 + col;
      unit_step = 64;
      half_step = KH * st;
      rows = extent - row0 - col;
      off0 = (uint32_t)(k * 128 + (((lane & 7) ^ (k & 7)) << 4));
    } else {
      const int r8 = ((lane >> 2) & 1) * 4 + (lane >> 3), r = warp * 8 + r8, u = lane & 3;
      kofs = u * 8;
      p = base + (long long)(row0 + r) * st + k0 + u * 8;
      unit_step = 64 * st;
      half_step = KH;
      rows = extent - row0 - r;
      off0 = (uint32_t)(r * 128 + ((u ^ r8) << 4));
    }
  }
  // odd slots hold k values 32..63 of the 64-deep swizzled rows
  __device__ __forceinline__ uint32_t off(int slot) const { return MN ? off0 + slot * 4096u : off0 ^ (slot * 64u); }   // slot 0 or 1
  // krem: k values left from the first one of the step
  __device__ __forceinline__ void fetch(float (&v)[UNITS][8], int krem) {
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      const float* q = p + i * unit_step;
      const int n = MN ? (kofs < krem ? rows - 64 * i : 0) : (64 * i < rows ? krem - kofs : 0);
      if (vec && n >= 8) {
        const float4 a = *reinterpret_cast<const float4*>(q), b = *(reinterpret_cast<const float4*>(q) + 1);
        v[i][0] = a.x; v[i][1] = a.y; v[i][2] = a.z; v[i][3] = a.w;
        v[i][4] = b.x; v[i][5] = b.y; v[i][6] = b.z; v[i][7] = b.w;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[i][e] = e < n ? q[e] : 0.f;
      }
    }
    p += half_step;
  }
  template <uint32_t PLANE, bool PACKED>
  __device__ __forceinline__ void store(const float (&v)[UNITS][8], uint8_t* plane0, int slot) const {
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      uint4 h, m, l;
      split2<PACKED>(v[i][0], v[i][1], h.x, m.x, l.x);
      split2<PACKED>(v[i][2], v[i][3], h.y, m.y, l.y);
      split2<PACKED>(v[i][4], v[i][5], h.z, m.z, l.z);
      split2<PACKED>(v[i][6], v[i][7], h.w, m.w, l.w);
      uint8_t* d = plane0 + off(slot) + i * 8192;
      *reinterpret_cast<uint4*>(d) = h;
      *reinterpret_cast<uint4*>(d + PLANE) = m;
      *reinterpret_cast<uint4*>(d + 2 * PLANE) = l;
    }
  }
};

// Slots of 32 k values (two to a swizzled row of 64): pairs have four, so that the relay's round trip
// between the CTAs is not waited for (with two: 512 x 16384 x 16384 8 % slower).
constexpr int slots_of(int pair) { return pair == 2 ? 4 : 2; }
template <int BN, int PAIR>
constexpr uint32_t ring_bytes() { return 3u * (BM + BN / PAIR) * 64u * slots_of(PAIR); }
// k values, rows and columns of redo(), and its operands in shared memory behind the finished tile
constexpr int kRedoK = 32, kRedoRows = 128, kRedoCols = 64;
constexpr int kRedoBytes = kRedoK * (kRedoRows + 4 + kRedoCols + 4) * 4;
template <int BN, int PAIR>
constexpr uint32_t smem_bytes() {
  const uint32_t tile = BM * (BN + 4) * 4 + kRedoBytes;
  return (ring_bytes<BN, PAIR>() > tile ? ring_bytes<BN, PAIR>() : tile) + 1024;
}

// Barrier of the kThreads threads that run finish(); returns whether `p` holds in any of them.
__device__ __forceinline__ bool finish_barrier(bool p) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred q, r;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.cta.red.or.pred r, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, r;\n\t}"
      : "=r"(any) : "r"((uint32_t)p), "n"(kThreads) : "memory");
  return any != 0;
}
__device__ __forceinline__ bool is_finite(float v) { return fabsf(v) <= FLT_MAX; }

// Four adjacent results through the epilogue.
__device__ __forceinline__ void emit(const F32Args& a, const F32Problem& pr, int g, int m, int n, float (&v)[4]) {
  const int cnt = min(4, pr.N - n);
  float* out = pr.out + (long long)g * pr.out_sg + (long long)m * pr.out_ld + n;
  const bool wide = (pr.vec & 4) && cnt == 4;
  float x[4] = {0.f, 0.f, 0.f, 0.f};                    // the epilogue's other input: bias, mask or the old weight
  const float* src = pr.epi == EPI_SGD ? out
                     : pr.epi == EPI_RELU_MASK ? pr.mask + (long long)g * pr.mask_sg + (long long)m * pr.mask_ld + n
                     : pr.bias                 ? pr.bias + (long long)g * pr.bias_sg + n : nullptr;
  if (src) {
    if (wide) {
      const float4 t = *reinterpret_cast<const float4*>(src);
      x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < cnt) x[u] = src[u];
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (pr.epi == EPI_SGD) v[u] = x[u] - a.lr * v[u];
    else if (pr.epi == EPI_RELU_MASK) v[u] = x[u] > 0.f ? v[u] : 0.f;
    else {
      v[u] += x[u];
      if (pr.epi == EPI_BIAS_RELU) v[u] = fmaxf(v[u], 0.f);
    }
  }
  if (wide) {
    *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < cnt) out[u] = v[u];
  }
}

// 128 rows x 64 columns from (r0, c0) of the tile once more, as chains of fp32 multiply-adds with k ascending:
// the results that finish() left behind because a sum of theirs is not finite.  32 k values at a time go
// through shared memory (`slab`), the next ones on their way; a thread forms 4 x 4 results.  The k loop ends
// when all of them are NaN.
// An evaluation of 512 rows on 256-2048-2048-2048 with one hidden neuron at infinity: 0.79 ms (0.13 with
// finite values, 12.8 with a chain per result and thread); on 1024-8192-8192-100 5.2 ms (0.44).
template <int A_MN, int B_MN, int PITCH>
__device__ __forceinline__ void redo(const F32Args& a, const F32Problem& pr, int g, int m0, int n0, int r0, int live, int c0,
                                     const float* tile_s, float* slab, int tid) {
  constexpr int PA = kRedoRows + 4, PB = kRedoCols + 4;  // rows stay 16-byte aligned
  constexpr int NA = kRedoRows * kRedoK / kThreads, NB = kRedoCols * kRedoK / kThreads;
  float* sa = slab;                                      // [kRedoK][PA]
  float* sb = slab + kRedoK * PA;                        // [kRedoK][PB]
  const int ty = tid / 16, tx = tid % 16;                // this thread's rows 4 ty.., columns 4 tx..
  const float* A = pr.A + (long long)g * pr.a_sg;
  const float* B = pr.B + (long long)g * pr.b_sg;
  float acc[4][4];
  uint32_t need = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[i][j] = 0.f;
      if (4 * ty + i < live && n0 + c0 + 4 * tx + j < pr.N && !is_finite(tile_s[(r0 + 4 * ty + i) * PITCH + c0 + 4 * tx + j]))
        need |= 1u << (4 * i + j);
    }
  const bool any_here = __any_sync(0xffffffffu, need != 0);   // in this warp's 8 rows
  float ra[NA], rb[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int e = tid + kThreads * u, k = k0 + (A_MN ? e / kRedoRows : e % kRedoK), m = A_MN ? e % kRedoRows : e / kRedoK;
      const long long row = m0 + r0 + m;
      ra[u] = m < live && k < pr.K ? A[A_MN ? k * pr.a_st + row : row * pr.a_st + k] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + kThreads * u, k = k0 + (B_MN ? e / kRedoCols : e % kRedoK), n = n0 + c0 + (B_MN ? e % kRedoCols : e / kRedoK);
      rb[u] = n < pr.N && k < pr.K ? B[B_MN ? k * pr.b_st + n : n * pr.b_st + k] : 0.f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < pr.K; k0 += kRedoK) {
    bool alive = false;                                  // a result that is not NaN yet
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) alive |= (need >> (4 * i + j) & 1) && acc[i][j] == acc[i][j];
    if (!finish_barrier(alive)) break;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int e = tid + kThreads * u;
      sa[(A_MN ? e / kRedoRows : e % kRedoK) * PA + (A_MN ? e % kRedoRows : e / kRedoK)] = ra[u];
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + kThreads * u;
      sb[(B_MN ? e / kRedoCols : e % kRedoK) * PB + (B_MN ? e % kRedoCols : e / kRedoK)] = rb[u];
    }
    finish_barrier(false);
    if (k0 + kRedoK < pr.K) fetch(k0 + kRedoK);
    if (!any_here) continue;
#pragma unroll 4
    for (int k = 0; k < kRedoK; ++k) {
      const float4 x = *reinterpret_cast<const float4*>(sa + k * PA + 4 * ty), y = *reinterpret_cast<const float4*>(sb + k * PB + 4 * tx);
      const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xs[i], ys[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!(need >> (4 * i) & 15)) continue;
    const int r = r0 + 4 * ty + i, c = c0 + 4 * tx;
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = need >> (4 * i + j) & 1 ? acc[i][j] : tile_s[r * PITCH + c + j];
    emit(a, pr, g, m0 + r, n0 + c, v);
  }
}

// Closing part of a tile, run by kThreads threads: the finished sums lie in shared memory, row by row;
// apply the epilogue to this CTA's share of the rows and write the result.
template <int A_MN, int B_MN, int BN, int PAIR>
__device__ __forceinline__ void finish(const F32Args& a, const F32Problem& pr, int g, int m0, int n0, int rank, int cluster,
                                       float* tile_s, int tid) {
  constexpr int PITCH = BN + 4, Q = BN / 4;             // Q 4-column pieces of a row
  const int share = PAIR == 1 ? BM / cluster : BM;      // rows this CTA finishes
  const int r_lo = PAIR == 1 ? rank * share : 0;
  const int live = min(share, pr.M - m0 - r_lo);        // those inside the result
  const uint32_t tile_u = smem_u32(tile_s);
  bool left = false;
#pragma unroll 2
  for (int e = tid; e < live * Q; e += kThreads) {
    const int r = r_lo + e / Q, c4 = (e % Q) * 4, m = m0 + r, n = n0 + c4;
    if (n >= pr.N) continue;
    float v[4];
    float4* mine = reinterpret_cast<float4*>(tile_s + r * PITCH + c4);
    if (PAIR == 1 && cluster > 1) {
      v[0] = v[1] = v[2] = v[3] = 0.f;
      for (int s = 0; s < cluster; ++s) {               // in rank order: a fixed sum
        uint32_t addr;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(tile_u + (uint32_t)(r * PITCH + c4) * 4), "r"(s));
        const float4 t = ld_cluster4(addr);
        v[0] += t.x; v[1] += t.y; v[2] += t.z; v[3] += t.w;
      }
    } else {
      const float4 t = *mine;
      v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
    bool ok = true;
#pragma unroll
    for (int u = 0; u < 4; ++u) ok &= is_finite(v[u]) || n + u >= pr.N;
    if (ok) {
      emit(a, pr, g, m, n, v);
    } else {                                            // nobody else reads these rows of this CTA's sums
      *mine = make_float4(v[0], v[1], v[2], v[3]);
      left = true;
    }
  }
  if (finish_barrier(left)) {
    float* slab = tile_s + BM * PITCH;
#pragma unroll 1
    for (int c0 = 0; c0 < BN && n0 + c0 < pr.N; c0 += kRedoCols)
      redo<A_MN, B_MN, PITCH>(a, pr, g, m0, n0, r_lo, live, c0, tile_s, slab, tid);
  }
}

template <int A_MN, int B_MN, int BN, int PAIR>
__global__ void __launch_bounds__(threads_of(BN), 1) gemm_f32_kernel(const __grid_constant__ F32Args a) {
  constexpr int BNL = BN / PAIR;                       // rows of B this CTA loads
  constexpr uint32_t A_BYTES = BM * 128, PLANE = A_BYTES + BNL * 128;
  constexpr int UA = BM / 64, UB = BNL / 64;
  constexpr int NACC = BN / 2;                         // sums per adding thread
  constexpr int PITCH = BN + 4;                        // floats per row of the finished tile in shared memory
  constexpr int DEPTH = BN == 256 ? 1 : 2;             // steps whose operands are on their way to registers
  constexpr int SLOTS = slots_of(PAIR), LG = SLOTS == 4 ? 2 : 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float* tile_s = reinterpret_cast<float*>(smem);
  __shared__ uint64_t full[SLOTS], done[SLOTS], taken[2], peer[SLOTS];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  constexpr bool WHOLE = BN != 256;                    // see issue
  const int tid = threadIdx.x, warp = WHOLE ? __shfl_sync(0xffffffffu, tid >> 5, 0) : tid >> 5, lane = tid & 31;
  const int cluster = PAIR == 2 ? 2 : a.ksplit;
  const int side = (int)blockIdx.x - a.p[a.n_problems - 1].tile_end * cluster;
  if (side >= 0) {                                     // bias work (a whole cluster of it)
    pdl_wait();
    pdl_trigger();
    for (int b = side; b < a.side_blocks; b += a.side_ctas) {
      bias_block(a.bias, b, tid, reinterpret_cast<float(*)[65]>(smem));
      __syncthreads();
    }
    return;
  }
  const int rank = cluster > 1 ? (int)cluster_ctarank() : 0;
  if (tid == 0) {
    for (int b = 0; b < SLOTS; ++b) {
      mbar_init(&full[b], kLoadWarps + (PAIR == 2 && rank == 0 ? 1 : 0));
      mbar_init(&done[b], 1);
      mbar_init(&peer[b], 1);
    }
    for (int b = 0; b < 2; ++b) mbar_init(&taken[b], PAIR * kAddWarps);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 0) {
    if (PAIR == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(2 * BN) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(2 * BN) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR == 2) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;

  // which tile, and which part of its k range
  int pi = 0, tile = (int)blockIdx.x / cluster;
  while (tile >= a.p[pi].tile_end) ++pi;
  const F32Problem& pr = a.p[pi];
  tile -= pi ? a.p[pi - 1].tile_end : 0;
  const int mt = tile % pr.m_tiles, rest = tile / pr.m_tiles, nt = rest % pr.n_tiles, g = rest / pr.n_tiles;
  const int m0 = mt * (BM * PAIR) + (PAIR == 2 ? rank * BM : 0);   // this CTA's rows of A and of the result
  const int n0 = nt * BN;                                          // first column of the tile
  int step0 = 0, steps = (pr.K + KH - 1) / KH;
  if (PAIR == 1 && cluster > 1) {
    const int per = (steps + cluster - 1) / cluster;
    step0 = min(rank * per, steps);
    steps = min(per, steps - step0);
  }

  pdl_wait();       // everything above touched this CTA's own memory only, see common.cuh
  pdl_trigger();

  // After the last MMA: sums into shared memory, tensor memory back, results out.  Both roles
  // come here by their own copy of the code, so that each keeps its own register allotment.
  auto close = [&](const uint64_t* acc) {
    tc_fence_before();
    __syncthreads();
    if (PAIR == 2) cluster_sync_all();   // the peer's MMAs have read this CTA's shared memory
    const bool bad = *abortp != 0;
    if (acc) {
      float* row = tile_s + ((warp & 3) * 32 + lane) * PITCH + ((warp - kLoadWarps) >> 2) * NACC;
#pragma unroll
      for (int c = 0; c < NACC / 4; ++c)
        *reinterpret_cast<ulonglong2*>(row + 4 * c) = make_ulonglong2(acc[2 * c], acc[2 * c + 1]);
    } else if (warp == 0) {
      __syncwarp();
      if (PAIR == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
      else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
    if (PAIR == 1 && cluster > 1) cluster_sync_all(); else __syncthreads();
    if (!bad && warp < kLoadWarps + kAddWarps) finish<A_MN, B_MN, BN, PAIR>(a, pr, g, m0, n0, rank, cluster, tile_s, tid);
    if (PAIR == 1 && cluster > 1) cluster_sync_all();   // the others have read this CTA's sums
  };

  // Descriptors of slot 0, plane 0; the others lie a constant further (an address in 16-byte
  // units, below 2^14).  Built afresh for every MMA they took 60 cycles each, more than the
  // tensor core's work on a 64-column tile.
  constexpr uint32_t idesc = make_idesc(A_MN, B_MN, BN, BM * PAIR);
  const uint64_t ad0 = A_MN ? make_desc(smem_u32(smem), 8192, 1024) : make_desc(smem_u32(smem), 16, 1024);
  const uint64_t bd0 = B_MN ? make_desc(smem_u32(smem) + A_BYTES, 8192, 1024) : make_desc(smem_u32(smem) + A_BYTES, 16, 1024);
  // The MMAs of step i.  Narrow tiles: the warp that has nothing else to do goes through this whole, one elected lane
  // issues (see elect_one; 784-1024-10, S = 2, 128 rows, ten steps 407 -> 393 us).  256 columns: one lane of an adding warp
  // does; with the whole warp in it, evaluation of 3072-16384-16384-10 takes 15.2 instead of 14.1 ms.
  auto issue = [&](int i, bool leader) -> bool {
    const int b = i & 1, sl = i & (SLOTS - 1);
    auto reached = [&](bool ok) { return WHOLE ? (bool)__all_sync(0xffffffffu, ok) : ok; };
    if (!reached(mbar_wait(&full[sl], (i >> LG) & 1, abortp, a.status, 21))) return false;
    if (i >= 2 && !reached(mbar_wait<PAIR == 2>(&taken[b], ((i >> 1) & 1) ^ 1, abortp, a.status, 23))) return false;
    tc_fence_after();
    constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};   // low x high first, high x high last
    const uint32_t at = (uint32_t)(sl >> 1) * (3 * PLANE >> 4);
    const uint64_t ad = ad0 + at + (b ? (A_MN ? 4096 : 64) >> 4 : 0), bd = bd0 + at + (b ? (B_MN ? 4096 : 64) >> 4 : 0);
    if (leader) {
#pragma unroll
      for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int k = 0; k < KH / 16; ++k) {
          const uint64_t da = ad + ((pa[c] * PLANE + k * (A_MN ? 2048 : 32)) >> 4);
          const uint64_t db = bd + ((pb[c] * PLANE + k * (B_MN ? 2048 : 32)) >> 4);
          if ((c == 3 || c == 5) && k == 0) {              // from one weight to the next: 2^8
            if (PAIR == 2) tc_mma_pair<8>(tmem + b * BN, da, db, idesc, 1);
            else tc_mma<8>(tmem + b * BN, da, db, idesc, 1);
          } else {
            if (PAIR == 2) tc_mma_pair(tmem + b * BN, da, db, idesc, (c | k) != 0);
            else tc_mma(tmem + b * BN, da, db, idesc, (c | k) != 0);
          }
        }
      if (PAIR == 2) tc_commit_pair(&done[sl]); else tc_commit(&done[sl]);
    }
    if (WHOLE) __syncwarp();
    return true;
  };
  // Pairs: passes on that the peer CTA's half of step i lies in its shared memory.
  auto relay = [&](int i) {
    if (i >= steps) return;
    const int sl = i & (SLOTS - 1);
    if (!mbar_wait<true>(rank ? &full[sl] : &peer[sl], (i >> LG) & 1, abortp, a.status, 24)) return;
    if (rank) mbar_arrive_cluster<true>(map_to_cta(&peer[sl], 0)); else mbar_arrive(&full[sl]);
  };

  if (warp < kLoadWarps) {
    // ---------------------------------------------------------------- load and split
    // registers at launch: 512 threads x 128, or 640 x 96
    if (BN == 256) asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    Operand<A_MN, UA> oa;
    Operand<B_MN, UB> ob;
    oa.init(pr.A + (long long)g * pr.a_sg, pr.a_st, m0, pr.M, step0 * KH, tid, pr.vec & 1);
    ob.init(pr.B + (long long)g * pr.b_sg, pr.b_st, n0 + (PAIR == 2 ? rank * BNL : 0), pr.N, step0 * KH, tid, pr.vec & 2);
    float va[DEPTH][UA][8], vb[DEPTH][UB][8];
    int krem = pr.K - step0 * KH;        // k values left from the next step to request
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) {
      if (d < steps) {
        oa.fetch(va[d], krem);
        ob.fetch(vb[d], krem);
      }
      krem -= KH;
    }
    bool ok = true;
    auto step = [&](int i, float (&xa)[UA][8], float (&xb)[UB][8]) {
      const int sl = i & (SLOTS - 1);
      if (i >= SLOTS) {
        ok = __all_sync(0xffffffffu, mbar_wait(&done[sl], ((i >> LG) & 1) ^ 1, abortp, a.status, 22));
        if (!ok) return;
      }
      uint8_t* slot = smem + (sl >> 1) * (3 * PLANE);
      oa.template store<PLANE, PAIR == 2>(xa, slot, sl & 1);
      ob.template store<PLANE, PAIR == 2>(xb, slot + A_BYTES, sl & 1);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[sl]);
      if (i + DEPTH < steps) {
        oa.fetch(xa, krem);
        ob.fetch(xb, krem);
        krem -= KH;
      }
    };
    for (int i = 0; i < steps && ok; i += DEPTH) {
#pragma unroll
      for (int d = 0; d < DEPTH; ++d)
        if (i + d < steps && ok) step(i + d, va[d], vb[d]);
    }
    close(nullptr);
  } else if (BN == 256 || warp < kLoadWarps + kAddWarps) {
    // ---------------------------------------------------------------- add up
    if (BN == 256) asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const bool issuer = BN == 256 && warp == kLoadWarps && lane == 0 && rank == 0;
    const bool relayer = PAIR == 2 && warp == kLoadWarps + 1 && lane == 0;
    constexpr int AHEAD = 2;                           // steps ahead of the one being added up, see above
    constexpr int W = BN == 256 ? 16 : 32;             // columns per tensor-memory load
    uint64_t acc[NACC / 2];
#pragma unroll
    for (int i = 0; i < NACC / 2; ++i) acc[i] = 0;
    const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(((warp - kLoadWarps) >> 2) * NACC);
    if (issuer && steps > 0) issue(0, true);
    if (relayer)
      for (int i = 0; i < AHEAD; ++i) relay(i);
    __syncwarp();
    for (int i = 0; i < steps; ++i) {
      const int b = i & 1;
      if (issuer && i + 1 < steps) issue(i + 1, true);
      if (relayer) relay(i + AHEAD);
      __syncwarp();
      if (!__all_sync(0xffffffffu, mbar_wait(&done[i & (SLOTS - 1)], (i >> LG) & 1, abortp, a.status, 20))) break;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < NACC; c += W) {
        uint32_t v[W];
        if (W == 32) tc_ld32(t_row + (uint32_t)(b * BN + c), v);
        else tc_ld16(t_row + (uint32_t)(b * BN + c), v);
#pragma unroll
        for (int e = 0; e < W / 2; ++e) add2(acc[c / 2 + e], v[2 * e], v[2 * e + 1]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR == 2) mbar_arrive_relaxed_cluster(map_to_cta(&taken[b], 0));
        else mbar_arrive(&taken[b]);
      }
    }
    close(acc);
  } else {
    // ---------------------------------------------------------------- issue the MMAs of a narrow tile
    asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
    if (warp == kLoadWarps + kAddWarps) {
      const bool leader = elect_one();
      for (int i = 0; i < steps; ++i)
        if (!issue(i, leader)) break;
    }
    __syncwarp();
    close(nullptr);
  }
}

// ---- host side ---------------------------------------------------------------------------------

template <int A_MN, int B_MN, int BN, int PAIR>
bool launch(const Launch& L, const F32Args& t, int cluster) {
  auto kern = gemm_f32_kernel<A_MN, B_MN, BN, PAIR>;
  constexpr int smem = (int)smem_bytes<BN, PAIR>();
  static bool ready = false;
  static std::once_flag once;
  std::call_once(once, [&] {
    ready = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
  });
  if (!ready) return false;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(t.p[t.n_problems - 1].tile_end * cluster + t.side_ctas));
  cfg.blockDim = dim3(threads_of(BN));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = L.stream;
  cudaLaunchAttribute attrs[2];
  int n = 0;
  attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attrs[n++].val.programmaticStreamSerializationAllowed = 1;
  if (cluster > 1) {
    attrs[n].id = cudaLaunchAttributeClusterDimension;
    attrs[n].val.clusterDim.x = (unsigned)cluster;
    attrs[n].val.clusterDim.y = 1;
    attrs[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attrs;
  cfg.numAttrs = n;
  if (cudaLaunchKernelEx(&cfg, kern, t) != cudaSuccess) return false;
  L.count();
  return true;
}

template <int A_MN, int B_MN>
bool launch_bn(const Launch& L, const F32Args& t, int bn, int pair, int cluster) {
  if (pair == 2) return launch<A_MN, B_MN, 256, 2>(L, t, 2);
  if (bn == 128) return launch<A_MN, B_MN, 128, 1>(L, t, cluster);
  return launch<A_MN, B_MN, 64, 1>(L, t, cluster);
}

// Clusters of two, four and eight CTAs that can run at once (a GPU processing cluster holds a whole
// number of them): 16 of eight did not all fit and took two rounds (128 x 512 x 784 of two groups, 64
// columns: 18.5 us in clusters of eight, 11.7 us in clusters of four).
int clusters_at_once(int cluster) {
  static int n[4] = {148, 0, 0, 0};
  static std::once_flag once;
  std::call_once(once, [] {
    auto kern = gemm_f32_kernel<0, 1, 128, 1>;           // the larger of the two single-CTA shapes
    constexpr int smem = (int)smem_bytes<128, 1>();
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return;
    for (int i = 1; i < 4; ++i) {
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(128);
      cfg.blockDim = dim3(threads_of(128));
      cfg.dynamicSmemBytes = smem;
      cudaLaunchAttribute attr{};
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = 1u << i;
      attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      int k = 0;
      if (cudaOccupancyMaxActiveClusters(&k, kern, &cfg) == cudaSuccess) n[i] = k;
    }
  });
  return n[cluster == 1 ? 0 : cluster == 2 ? 1 : cluster == 4 ? 2 : 3];
}

// Tile shape and k split of a launch, and its estimated time in microseconds: as many rounds of
// tiles as the SMs need, each a fixed part (start, first operands, epilogue) and so much per
// 32-deep step.  Constants fitted to 12 products of 64 x 64 x 32 to 512 x 16384 x 3072 (measured
// 5.3 to 244 us, estimates within 25 %); 64-column tiles pay off only where 128-column ones leave
// SMs idle or the product is narrow, pairs from about 64 tiles of 256 x 256 on.
struct Shape { int bn, pair, cluster; double us; };
Shape pick_shape(const GemmArgs<float>* ga, int n) {
  const int sms = 148;
  Shape best{64, 1, 1, 1e300};
  auto consider = [&](int bn, int pair, int cluster, double step_us, double fix_us) {
    int64_t tiles = 0, steps = 0;
    for (int i = 0; i < n; ++i) {
      tiles += ceil_div(ga[i].M, BM * pair) * ceil_div(ga[i].N, bn) * ga[i].G;
      steps = std::max<int64_t>(steps, ceil_div(ga[i].K, KH));
    }
    if (cluster > 1 && (steps < 2 * cluster || tiles > clusters_at_once(cluster))) return;
    const int64_t rounds = ceil_div(tiles * pair, sms);
    const double us = rounds * (fix_us + step_us * ceil_div(steps, cluster)) + (cluster > 1 ? 0.5 + 0.2 * cluster : 0.0);
    if (us < best.us) best = Shape{bn, pair, cluster, us};
  };
  for (int cl = 1; cl <= 8; cl *= 2) {
    consider(64, 1, cl, 0.95, 4.0);
    consider(128, 1, cl, 1.2, 5.0);
  }
  consider(256, 2, 1, 1.15, 13.0);
  return best;
}

// Whether the CUDA-core kernel for short contractions is the quicker one: always up to 16 k values
// (half a step here; 256 x 1024 x 16 of four groups 6.1 against 7.6 us), else by its time as
// measured, 3 us and (1.4 + 0.1 K) us per 1024 tiles of 32 x 32 (64 x 64 x 64 of four groups 3.5
// against 6.2 us, 512 x 4096 x 64 19 against 12 us).
bool short_wins(const GemmArgs<float>* a, int n, double us) {
  double mine = 3.0;
  bool half = true;
  for (int i = 0; i < n; ++i) {
    if (a[i].K > 64) return false;
    half &= a[i].K <= 16;
    mine += (1.4 + 0.1 * a[i].K) * (double)ceil_div(a[i].M, 32) * ceil_div(a[i].N, 32) * a[i].G / 1024;
  }
  return half || mine < us;
}

}  // namespace

bool gemm_f32(const Launch& L, const GemmArgs<float>* ga, int n, const BiasSgdArgs<float>* bias, DeviceStatus* st) {
  if (n < 1 || n > kMaxProblems) return false;
  // One layout per operand for the whole launch: contiguous along k, or along m / n.  An operand with unit
  // stride in both directions (a width of one) fits either and goes with the others.
  bool a_k = true, a_m = true, b_k = true, b_n = true;
  for (int i = 0; i < n; ++i) {
    const GemmArgs<float>& a = ga[i];
    if (a.M < 1 || a.N < 1 || a.K < 1 || a.G < 1 || a.lr != ga[0].lr) return false;
    a_k &= a.a_sk == 1; a_m &= a.a_sm == 1;
    b_k &= a.b_sk == 1; b_n &= a.b_sn == 1;
  }
  if ((!a_k && !a_m) || (!b_k && !b_n)) return false;
  const bool a_mn = !a_k, b_mn = !b_k || (a_mn && b_n);
  const Shape sh = pick_shape(ga, n);
  if (short_wins(ga, n, sh.us) && gemm_short(L, ga, n, bias)) return true;
  F32Args t{};
  t.n_problems = n;
  t.ksplit = sh.cluster;
  t.lr = ga[0].lr;
  t.status = st;
  int64_t end = 0;
  for (int i = 0; i < n; ++i) {
    const GemmArgs<float>& a = ga[i];
    F32Problem& p = t.p[i];
    p.M = a.M; p.N = a.N; p.K = a.K; p.G = a.G;
    const int64_t mt = ceil_div(a.M, BM * sh.pair), nt = ceil_div(a.N, sh.bn);
    p.m_tiles = (int)mt;
    p.n_tiles = (int)nt;
    end += mt * nt * a.G;
    if (end * 8 > 0x7fffffffll) return false;
    p.tile_end = (int)end;
    p.epi = a.epi;
    p.A = a.A; p.a_st = a_mn ? a.a_sk : a.a_sm; p.a_sg = a.a_sg;
    p.B = a.B; p.b_st = b_mn ? a.b_sk : a.b_sn; p.b_sg = a.b_sg;
    const bool f32_out = a.epi == EPI_SGD || a.epi == EPI_BIAS_F32;
    p.bias = (a.epi == EPI_BIAS_RELU || a.epi == EPI_BIAS_F32) ? a.bias : nullptr; p.bias_sg = a.bias_sg;
    p.out = f32_out ? a.outf : a.out;
    p.out_ld = f32_out ? a.outf_ld : a.out_ld;
    p.out_sg = f32_out ? a.outf_sg : a.out_sg;
    p.mask = a.mask; p.mask_ld = a.mask_ld; p.mask_sg = a.mask_sg;
    auto vec = [](const void* q, int64_t ld, int64_t sg) { return ((uintptr_t)q & 15) == 0 && ld % 4 == 0 && sg % 4 == 0; };
    if (vec(p.A, p.a_st, p.a_sg)) p.vec |= 1;
    if (vec(p.B, p.b_st, p.b_sg)) p.vec |= 2;
    if (vec(p.out, p.out_ld, p.out_sg) && (!p.bias || vec(p.bias, 0, p.bias_sg)) &&
        (a.epi != EPI_RELU_MASK || vec(p.mask, p.mask_ld, p.mask_sg)))
      p.vec |= 4;
  }
  if (bias) {
    // one CTA per block of bias work, but no more than a round of them
    t.bias = *bias;
    t.side_blocks = bias_blocks(t.bias);
    const int cl = sh.pair == 2 ? 2 : sh.cluster;
    t.side_ctas = (int)ceil_div(std::min(t.side_blocks, 148), cl) * cl;
  }
  if (a_mn && b_mn) return launch_bn<1, 1>(L, t, sh.bn, sh.pair, sh.cluster);
  if (!a_mn && b_mn) return launch_bn<0, 1>(L, t, sh.bn, sh.pair, sh.cluster);
  if (!a_mn) return launch_bn<0, 0>(L, t, sh.bn, sh.pair, sh.cluster);
  return false;
}

}  // namespace ist
