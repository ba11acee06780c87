// Second pass over a very wide output layer behind a narrow hidden layer (paper Sec. 2.1 "Training Subnets" on the
// slice W_t[G^s, :]), everything that follows the rows' log-sum-exp in one kernel.  Per block of 64 classes:
//
//   z = x W + b,  delta = (softmax - onehot) / B   (bf16, stays in shared memory)
//   dx += delta W^T                                (tensor memory, 160 blocks at most; one partial sum per CTA and subnet)
//   W -= lr x^T delta,  b -= lr sum_b delta        (the weights as they stood before the step are read first)
//
// What bounds it: the weights, 4 bytes per weight (operand and low half, see join_master) in and out.  As separate launches
// the deltas of 670,091 classes (2.7 GB per step at 256 rows and S = 8) were written once and read twice beside
// them and the operands were read three times.  135909-1024-670091, S = 8, 256 rows, per step: softmax and delta 1.10 ms,
// dx 0.72, update 1.73; in this pass 1.77, 0.47 of the copy rate on its 5.5 GB (1.50 with three shortcuts that lost precision:
// bias sums on mma.sync, dx of all of a CTA's classes in one sum, no tie bits).  What is left is the chain of a block's
// hand-offs (z, delta, products, bias sums, update, store: some 18,000 cycles from load to reload, five blocks in flight).
//
// Layout.  The subnet's x (256 rows x 128 neurons, 64 KB) stays in shared memory; a block's operands and low halves are
// [neuron][64 classes] tiles of 128-byte rows, five and three of them in flight; delta is [row][64 classes].  All three are
// 128-byte swizzled and each serves both products it takes part in, once K-major and once MN-major.  64 classes because
// tensor memory holds dx (2 x 128 columns), z (2 x 64) and two accumulators of the weight gradient (2 x 64), 512 in all.
// Products of 64 columns read shared memory faster than it delivers (48 instead of 32 cycles each): 2050 cycles of
// the tensor pipe per block, against 2900 for its 64 KB of DRAM traffic.
//
// Warps: 0 copies; 1-2 MMA issue; 3-18 z -> delta, eight per 128 rows, 32 columns of one row per thread (with eight
// warps and 64 columns the chain z -> delta was the longest: by 0.06 ms); 19-26 column sums of delta (bias) and weight
// updates, two groups of four that take turns; 27 stores and loads of the low halves.  All hand-offs are mbarriers, every wait
// is bounded, no CTA waits for another.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "tc_ptx.cuh"
#include "tma_map.h"

namespace ist {
namespace {

constexpr int kCols = 64;                 // classes of a block
constexpr int kStages = 4;                // of the first pass
constexpr int kHi = 5, kLo = 3;           // tiles of operands and of low halves in flight
constexpr int kThreads = 28 * 32;
constexpr uint32_t kXChunk = 256 * 128;   // 64 neurons of 256 rows
constexpr uint32_t kXBytes = 2 * kXChunk, kDeltaBytes = 256 * 128, kTile = 128 * 128;
constexpr int kSmem = kXBytes + kDeltaBytes + (kHi + kLo) * kTile + 1024;
// Blocks whose share of dx is summed in tensor memory, at most: 10,240 classes.  Sums there lose precision with their
// length, and slices of the separate launches have some 10,500.
constexpr int kDxBlocks = 160;
constexpr uint32_t kDxCol = 0, kZCol = 256, kDwCol = 384;

struct HeadArgs {
  int S, B, H, N, n_cta, blocks;         // blocks per subnet
  int ldw;                               // row length of the weights and biases
  int ldx;                               // row length of x, of dx partials and of the delta below
  int halves;                            // row blocks of 128
  int partials;                          // dx slabs per subnet
  float lr, inv_rows;
  const float* lse; const int32_t* labels; float* label_logit; long long lse_sg, labels_sg;
  float* bias; long long bias_sg;
  uint32_t* ties;                        // the masters' tie bits, see tie_bit
  float* dx_part;                        // [S][partials][B][ldx]
  float2* lse_part;                      // first pass: [S][partials][B] (reference exponent, sum)
  DeviceStatus* status;
};
struct HeadMaps {
  CUtensorMap x, hi, lo;
};

// Items (subnet, block) are numbered subnet by subnet; CTA i works on items [first_item(i), first_item(i + 1)).
__host__ __device__ __forceinline__ long long first_item(long long items, int n_cta, int i) { return items * i / n_cta; }
__host__ __device__ __forceinline__ int cta_of(long long items, int n_cta, long long item) {
  return (int)(((item + 1) * n_cta - 1) / items);
}

// Two fp32 operations in one instruction, each rounded as by itself.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// 16-byte unit u of 128-byte row r, 128-byte swizzled
__device__ __forceinline__ uint4* unit_at(uint8_t* tile, int r, int u) {
  return reinterpret_cast<uint4*>(tile + r * 128 + ((u ^ (r & 7)) << 4));
}

__global__ void __launch_bounds__(kThreads, 1)
wide_head_kernel(const __grid_constant__ HeadMaps maps, const __grid_constant__ HeadArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* x_s = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* delta_s = x_s + kXBytes;
  uint8_t* his = delta_s + kDeltaBytes;
  uint8_t* los = his + kHi * kTile;
  __shared__ uint64_t x_full, hi_full[kHi], hi_empty[kHi], lo_full[kLo], upd_done[kLo];
  __shared__ uint64_t z_full[2], z_empty[2], d_full[2], d_ready[2], d_empty[2], dw_full[2], dw_empty[2], dx_done, dx_flushed, x_free;
  __shared__ __align__(16) float bias_s[kHi][kCols];   // the block's biases travel with its operands
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: known to be uniform
  const int NH = a.halves;

  if (threadIdx.x == 0) {
    mbar_init(&x_full, 1);
    for (int s = 0; s < kHi; ++s) {
      mbar_init(&hi_full[s], 1);
      mbar_init(&hi_empty[s], 1);
    }
    for (int s = 0; s < kLo; ++s) {
      mbar_init(&lo_full[s], 1);
      mbar_init(&upd_done[s], 4);            // one per low-half tile: a block's has no second phase before its own store
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&z_full[h], 1);
      mbar_init(&z_empty[h], 8);
      mbar_init(&d_full[h], 8);
      mbar_init(&d_ready[h], 8 * NH);        // both halves of every other block's delta, for the group that sums it
      mbar_init(&d_empty[h], 1 + 4);         // the products' commit and the four summing warps
      mbar_init(&dw_full[h], 1);
      mbar_init(&dw_empty[h], 4);
    }
    mbar_init(&dx_done, 1);
    mbar_init(&dx_flushed, 8 * NH);
    mbar_init(&x_free, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (threadIdx.x == 32) {
    prefetch_map(&maps.x);
    prefetch_map(&maps.hi);
    prefetch_map(&maps.lo);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;
  pdl_wait();
  pdl_trigger();

  const long long items = (long long)a.S * a.blocks;
  const long long it0 = first_item(items, a.n_cta, blockIdx.x), it1 = first_item(items, a.n_cta, blockIdx.x + 1);
  const int count = (int)(it1 - it0);
  const int g0 = (int)(it0 / a.blocks), b0 = (int)(it0 - (long long)g0 * a.blocks);   // first subnet and block

  if (warp == 0) {
    // ---------------------------------------------------------------- loads of x, operands and biases
    if (lane == 0) {
      bool ok = true;
      int g = g0, blk = b0, groups = 0, i = 0;
      for (; i < count; ++i) {
        if (i == 0 || blk == 0) {
          // x of the next subnet: once every product that read the last one has completed
          if (groups > 0) ok = mbar_wait(&x_free, (groups - 1) & 1, abortp, a.status, 201);
          if (!ok) break;
          mbar_expect_tx(&x_full, kXBytes);
          tma_load_3d(x_s, &maps.x, &x_full, 0, 0, g);
          tma_load_3d(x_s + kXChunk, &maps.x, &x_full, 64, 0, g);
          ++groups;
        }
        const int s = i % kHi;
        ok = mbar_wait(&hi_empty[s], ((i / kHi) & 1) ^ 1, abortp, a.status, 202);
        if (!ok) break;
        const uint32_t bias_bytes = (uint32_t)min(kCols, a.ldw - blk * kCols) * 4;   // rows are padded to 32 bytes
        mbar_expect_tx(&hi_full[s], kTile + bias_bytes);
        bulk_load(bias_s[s], a.bias + g * a.bias_sg + blk * kCols, bias_bytes, &hi_full[s]);
        tma_load_3d(his + s * kTile, &maps.hi, &hi_full[s], blk * kCols, 0, g);
        if (++blk == a.blocks) { blk = 0; ++g; }
      }
      if (!ok) {   // copies in flight land before the CTA's shared memory goes away
        for (int j = max(0, i - kHi); j < i; ++j) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&hi_full[j % kHi], (j / kHi) & 1) && clock64() - t0 < kWaitLimitCycles) {}
        }
        const long long t0 = clock64();
        while (groups > 0 && !mbar_try_wait(&x_full, (groups - 1) & 1) && clock64() - t0 < kWaitLimitCycles) {}
      }
    }
  } else if (warp == 27) {
    // ---------------------------------------------------------------- stores, and loads of the low halves
    // One thread stores a block's updated tiles and then loads the low halves that take the place of its own; they are
    // wanted later than the operands and for a shorter time, so fewer of them are in flight.
    if (lane == 0) {
      bool ok = true;
      int g = g0, blk = b0, gs = g0, bs = b0, i = 0;   // block of the next load, of the next store
      auto store = [&](int j) -> bool {
        if (!mbar_wait(&upd_done[j % kLo], (j / kLo) & 1, abortp, a.status, 214)) return false;
        tma_store_3d(&maps.hi, his + (j % kHi) * kTile, bs * kCols, 0, gs);
        tma_store_3d(&maps.lo, los + (j % kLo) * kTile, bs * kCols, 0, gs);
        tma_commit_group();
        tma_wait_read<0>();
        mbar_arrive(&hi_empty[j % kHi]);
        if (++bs == a.blocks) { bs = 0; ++gs; }
        return true;
      };
      for (; i < count; ++i) {
        if (i >= kLo) ok = store(i - kLo);
        if (!ok) break;
        mbar_expect_tx(&lo_full[i % kLo], kTile);
        tma_load_3d(los + (i % kLo) * kTile, &maps.lo, &lo_full[i % kLo], blk * kCols, 0, g);
        if (++blk == a.blocks) { blk = 0; ++g; }
      }
      for (int j = max(0, count - kLo); j < count && ok; ++j) ok = store(j);
      tma_wait_all();
      if (!ok)
        for (int j = max(0, i - kLo); j < i; ++j) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&lo_full[j % kLo], (j / kLo) & 1) && clock64() - t0 < kWaitLimitCycles) {}
        }
    }
  } else if (warp <= 2) {
    // ---------------------------------------------------------------- products
    // Two warps issue, one z and the other dx and the weight gradient, so that one's products run while the other looks
    // at its barriers (some 300 cycles each time; with one warp the tensor pipe stood still for half of the time).
    // The whole warp runs this, one elected lane issues: descriptors then stay in uniform registers, and a product of 64
    // columns costs less to issue than to run (in a branch of one lane: 76 to 100 cycles each).
    const bool leader = elect_one();
    auto wait = [&](uint64_t* bar, uint32_t parity, int where) {
      return (bool)__all_sync(0xffffffffu, mbar_wait(bar, parity, abortp, a.status, where));
    };
    const int kz = (a.H + 15) / 16;                                // 16-deep steps of x W
    bool ok = true;
    int blk = b0;
    // descriptors of the tiles' first steps; the address field counts 16-byte units, so steps are additions
    if (warp == 1) {
      const uint32_t id_z = make_idesc(0, 1, kCols, 128);
      int groups = 0;
      bool fresh = true;                                           // first block of a subnet
      const uint64_t x_k = make_desc(smem_u32(x_s), 16, 1024), w0 = make_desc(smem_u32(his), 8192, 1024);
      for (int i = 0; i < count && ok; ++i) {
        if (fresh) ok = wait(&x_full, groups & 1, 205);
        const int s = i % kHi;
        ok = ok && wait(&hi_full[s], (i / kHi) & 1, 203);
        const uint64_t w = w0 + (uint64_t)((s * kTile) >> 4);
        for (int h = 0; h < NH && ok; ++h) {
          ok = wait(&z_empty[h], (i & 1) ^ 1, 204);
          if (!ok) break;
          tc_fence_after();
          const uint64_t x = x_k + (uint64_t)(h * 16384 >> 4);
          if (leader) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (k < kz)
                tc_mma(tmem + kZCol + h * kCols, x + (((k >> 2) * kXChunk + (k & 3) * 32) >> 4), w + (k * 2048 >> 4), id_z, k != 0);
            tc_commit(&z_full[h]);
          }
          __syncwarp();
        }
        fresh = blk + 1 == a.blocks;
        if (fresh) ++groups;
        if (++blk == a.blocks) blk = 0;
      }
    } else {
      const uint32_t id_dw = make_idesc(1, 1, kCols, 128), id_dx = make_idesc(0, 0, kz * 16, 128);
      const uint64_t x_mn = make_desc(smem_u32(x_s), kXChunk, 1024), w0 = make_desc(smem_u32(his), 16, 1024);
      const uint64_t d_k = make_desc(smem_u32(delta_s), 16, 1024), d_mn = make_desc(smem_u32(delta_s), 8192, 1024);
      int held = 0, parts = 0;                                     // blocks in dx so far; sums handed over
      for (int i = 0; i < count && ok; ++i) {
        if (held == 0 && parts > 0) ok = wait(&dx_flushed, (parts - 1) & 1, 206);
        const bool last = i + 1 == count || blk + 1 == a.blocks;   // of this subnet here
        const bool full = last || held + 1 == kDxBlocks;
        const uint64_t w = w0 + (uint64_t)(((i % kHi) * kTile) >> 4);
        const uint32_t dw = tmem + kDwCol + (i & 1) * kCols;
        ok = ok && wait(&dw_empty[i & 1], ((i >> 1) & 1) ^ 1, 207);
        for (int h = 0; h < NH && ok; ++h) {
          ok = wait(&d_full[h], i & 1, 208);
          if (!ok) break;
          tc_fence_after();
          const uint64_t dk = d_k + (uint64_t)(h * 16384 >> 4), dm = d_mn + (uint64_t)(h * 16384 >> 4);
          const uint64_t xm = x_mn + (uint64_t)(h * 16384 >> 4);
          if (leader) {
#pragma unroll
            for (int k = 0; k < kCols / 16; ++k)                   // dx[rows of h] += delta W^T
              tc_mma(tmem + kDxCol + h * 128, dk + (k * 32 >> 4), w + (k * 32 >> 4), id_dx, (held | k) != 0);
#pragma unroll
            for (int k = 0; k < 8; ++k)                            // x^T delta over the rows of h
              tc_mma(dw, xm + (k * 2048 >> 4), dm + (k * 2048 >> 4), id_dw, (h | k) != 0);
            tc_commit(&d_empty[h]);
          }
          __syncwarp();
        }
        if (!ok) break;
        if (leader) {
          tc_commit(&dw_full[i & 1]);
          if (full) tc_commit(&dx_done);
          if (last) tc_commit(&x_free);      // z of this block has completed too: delta was made from it
        }
        __syncwarp();
        held = full ? 0 : held + 1;
        if (full) ++parts;
        if (++blk == a.blocks) blk = 0;
      }
    }
  } else if (warp < 19) {
    // ---------------------------------------------------------------- z -> delta, and dx out at a subnet's end
    const int h = (warp - 3) >> 3, part32 = ((warp - 3) >> 2) & 1, q = warp & 3;   // 32 columns of a block
    const int r = q * 32 + lane, row = h * 128 + r;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    constexpr float kLog2e = 1.4426950408889634f;
    const bool live = row < a.B;
    bool ok = h < NH;
    int g = g0, blk = b0, held = 0, parts = 0;
    bool more = false;                       // dx of this subnet has been written before
    float row_lse = INFINITY;                // rows beyond the batch: delta is zero
    int label = -1;
    for (int i = 0; i < count && ok; ++i) {
      if ((i == 0 || blk == 0) && live) {
        row_lse = a.lse[g * a.lse_sg + row] * kLog2e - log2f(a.inv_rows);
        label = a.labels[g * a.labels_sg + row];
      }
      const int n0 = blk * kCols + 32 * part32;
      const float* bias = bias_s[i % kHi] + 32 * part32;
      // hi_full: the stage's copies have landed (the product waited for them), seen from this thread too for the biases
      ok = mbar_wait(&z_full[h], i & 1, abortp, a.status, 209) &&
           mbar_wait(&hi_full[i % kHi], (i / kHi) & 1, abortp, a.status, 216);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      uint32_t acc[32];
      tc_ld32(tmem + kZCol + h * kCols + 32 * part32 + lane_base, acc);
      tc_fence_before();                     // z is in registers: the next block's may follow
      __syncwarp();
      if (lane == 0) mbar_arrive(&z_empty[h]);
      uint4 o[4];                            // delta: kept until the last one has been read
      const int lat = label - n0;            // the label's column, if it is among these
      float zl = 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {          // 8 columns
        float z[8];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const float4 bv = *reinterpret_cast<const float4*>(bias + 8 * u + 4 * v);
          z[4 * v + 0] = __uint_as_float(acc[8 * u + 4 * v + 0]) + bv.x;
          z[4 * v + 1] = __uint_as_float(acc[8 * u + 4 * v + 1]) + bv.y;
          z[4 * v + 2] = __uint_as_float(acc[8 * u + 4 * v + 2]) + bv.z;
          z[4 * v + 3] = __uint_as_float(acc[8 * u + 4 * v + 3]) + bv.w;
        }
        uint32_t p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __nv_bfloat162 v = __floats2bfloat162_rn(ex2_approx(fmaf(z[2 * e], kLog2e, -row_lse)),
                                                         ex2_approx(fmaf(z[2 * e + 1], kLog2e, -row_lse)));
          p[e] = *reinterpret_cast<const uint32_t*>(&v);
        }
        o[u] = make_uint4(p[0], p[1], p[2], p[3]);
        if ((lat >> 3) == u)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if ((lat & 7) == e) zl = z[e];
      }
      if (n0 + 32 > a.N) {                   // the ragged block: its columns beyond the classes have no bias and no delta
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t* p = reinterpret_cast<uint32_t*>(&o[u]);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n = n0 + 8 * u + 2 * e;
            p[e] &= n + 1 < a.N ? 0xffffffffu : n < a.N ? 0xffffu : 0u;
          }
        }
      }
      __syncwarp();
      // the products of the block before have read the last delta of these rows
      ok = __all_sync(0xffffffffu, mbar_wait(&d_empty[h], (i & 1) ^ 1, abortp, a.status, 210));
      if (!ok) break;
#pragma unroll
      for (int u = 0; u < 4; ++u) *unit_at(delta_s, row, 4 * part32 + u) = o[u];
      if (lat >= 0 && lat < 32) {
        reinterpret_cast<bf16*>(unit_at(delta_s, row, 4 * part32 + (lat >> 3)))[lat & 7] =
            __float2bfloat16_rn(ex2_approx(fmaf(zl, kLog2e, -row_lse)) - a.inv_rows);
        a.label_logit[g * a.lse_sg + row] = zl;
      }
      __syncwarp();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&d_full[h]);
        mbar_arrive(&d_ready[i & 1]);
      }
      const bool last = i + 1 == count || blk + 1 == a.blocks;
      ++held;
      if (last || held == kDxBlocks) {
        // the subnet's last block here, or as many as are summed in one piece: their share of dx leaves tensor memory
        ok = __all_sync(0xffffffffu, mbar_wait(&dx_done, parts & 1, abortp, a.status, 211));
        if (!ok) break;
        tc_fence_after();
        const int part = (int)blockIdx.x - cta_of(items, a.n_cta, (long long)g * a.blocks);
        float* out = a.dx_part + (((long long)g * a.partials + part) * a.B + row) * a.ldx;
#pragma unroll 1
        for (int c = 2 * part32; c < 2 * part32 + 2; ++c) {
          if (32 * c >= a.ldx) break;
          uint32_t v[32];
          tc_ld32(tmem + kDxCol + h * 128 + c * 32 + lane_base, v);
          if (live)
#pragma unroll
            for (int u0 = 0; u0 < 8; u0 += 4) {      // four loads in flight
              float4 s[4];
#pragma unroll
              for (int u = 0; u < 4; ++u)
                s[u] = more && 32 * c + 4 * (u0 + u) < a.ldx ? *reinterpret_cast<const float4*>(out + 32 * c + 4 * (u0 + u))
                                                             : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const uint32_t* d = v + 4 * (u0 + u);
                if (32 * c + 4 * (u0 + u) < a.ldx)
                  *reinterpret_cast<float4*>(out + 32 * c + 4 * (u0 + u)) =
                      make_float4(s[u].x + __uint_as_float(d[0]), s[u].y + __uint_as_float(d[1]), s[u].z + __uint_as_float(d[2]),
                                  s[u].w + __uint_as_float(d[3]));
              }
            }
          __syncwarp();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dx_flushed);
        ++parts;
        held = 0;
        more = !last;
      }
      if (++blk == a.blocks) { blk = 0; ++g; }
    }
  } else {
    // ---------------------------------------------------------------- bias and weight updates
    const int grp = (warp - 19) >> 2, q = warp & 3;
    const int r = q * 32 + lane;             // neuron of this thread
    bool ok = true;
    const int chunks = (a.ldw + 31) / 32;
    auto has_ties = [&](int blk, int c) { return r < a.H && 2 * blk + c < chunks; };
    auto tie_word = [&](int g, int blk, int c) { return a.ties + ((long long)g * chunks + 2 * blk + c) * a.H + r; };
    for (int i = grp; i < count && ok; i += 2) {
      const int s = i % kHi;
      const int g = (int)((it0 + i) / a.blocks), blk = (int)(it0 + i - (long long)g * a.blocks);
      // tie bits: asked for here, the waits below take longer
      const uint32_t ties0 = has_ties(blk, 0) ? __ldcg(tie_word(g, blk, 0)) : 0u;
      const uint32_t ties1 = has_ties(blk, 1) ? __ldcg(tie_word(g, blk, 1)) : 0u;
      // Column sums of delta, 16 columns per warp: a lane adds up eight columns of every sixteenth row (the eight lanes of a
      // quarter warp read eight rows, every bank once), sixteen lanes then share their sums out.  All in fp32 additions: a row
      // of ones times delta on the tensor cores, accumulated from 16 rows to the next, was 6e-7 off over 256 rows
      // where additions in four chains are 0.8e-7 off, and always to the same side.
      ok = __all_sync(0xffffffffu, mbar_wait(&d_ready[grp], (i >> 1) & 1, abortp, a.status, 215));
      if (!ok) break;
      float c[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int h = 0; h < NH; ++h) {
        uint4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = *unit_at(delta_s, h * 128 + 16 * j + (lane & 15), 2 * q + (lane >> 4));
        __syncwarp();
        if (lane == 0) mbar_arrive(&d_empty[h]);   // these rows are in registers
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
                : "+f"(c[2 * e]), "+f"(c[2 * e + 1]) : "r"(w[e]));
        }
      }
      {
#pragma unroll
        for (int w = 4; w >= 1; w >>= 1) {   // of the columns held, a lane keeps half and gives the other half away
          const bool up = lane & (2 * w);
#pragma unroll
          for (int e = 0; e < w; ++e) {
            const float mine = up ? c[w + e] : c[e], other = up ? c[e] : c[w + e];
            c[e] = mine + __shfl_xor_sync(0xffffffffu, other, 2 * w);
          }
        }
        c[0] += __shfl_xor_sync(0xffffffffu, c[0], 1);
        const int col = 16 * q + 8 * (lane >> 4) + ((lane >> 1) & 7), n = blk * kCols + col;
        if ((lane & 1) == 0 && n < a.N) a.bias[g * a.bias_sg + n] = bias_s[s][col] - a.lr * c[0];
      }
      __syncwarp();
      ok = mbar_wait(&dw_full[grp], (i >> 1) & 1, abortp, a.status, 212) &&
           mbar_wait(&hi_full[s], (i / kHi) & 1, abortp, a.status, 213) &&
           mbar_wait(&lo_full[i % kLo], (i / kLo) & 1, abortp, a.status, 217);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      uint8_t* hi = his + s * kTile;
      uint8_t* lo = los + (i % kLo) * kTile;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        const uint32_t was = c ? ties1 : ties0;
        const uint32_t now = update_split32(tmem + kDwCol + grp * kCols + c * 32 + ((uint32_t)(q * 32) << 16), a.lr,
                                            [&](int u) { return unit_at(hi, r, 4 * c + u); },
                                            [&](int u) { return unit_at(lo, r, 4 * c + u); }, was, [&] {
                                              if (c == 0) return;
                                              tc_fence_before();
                                              __syncwarp();
                                              if (lane == 0) mbar_arrive(&dw_empty[grp]);
                                            });
        if (was | now)
          if (has_ties(blk, c)) *tie_word(g, blk, c) = now;
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&upd_done[i % kLo]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// First pass: the log-sum-exp of z = x W + b per row, z itself staying in tensor memory.  What bounds it is the special
// function unit, an ex2 per class and row (16 per clock and SM: 0.31 ms for 8 x 256 rows of 670,091 classes; the operands'
// 1.4 GB take 0.21).  Blocks of 128 classes, z double-buffered (2 x 2 x 128 columns), sixteen epilogue warps: warp
// group (h, p) takes rows 128 h .. + 127 and columns 64 p .. + 63 of every block.  A thread keeps its row's sum from
// the subnet's first block to its last, so a subnet has two partials per row and CTA.  The biases come through shared
// memory beside the operands: read from global memory, they were most of an epilogue's time.
// 135909-1024-670091, S = 8, 256 rows: 0.92 ms with the general kernel and its 10,472 partials per row, 0.53 here.
constexpr int kLseCols = 128;
constexpr int kLseThreads = 18 * 32;
constexpr uint32_t kLseStage = 2 * kTile;   // two boxes of 64 classes
constexpr int kLseSmem = kXBytes + kStages * kLseStage + 1024;

__global__ void __launch_bounds__(kLseThreads, 1)
wide_lse_kernel(const __grid_constant__ HeadMaps maps, const __grid_constant__ HeadArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* x_s = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* stages = x_s + kXBytes;
  __shared__ uint64_t x_full, w_full[kStages], w_empty[kStages], z_full[2][2], z_empty[2][2], grp_done;
  __shared__ __align__(16) float bias_s[kStages][kLseCols];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int NH = a.halves;

  if (threadIdx.x == 0) {
    mbar_init(&x_full, 1);
    mbar_init(&grp_done, 1);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&w_full[s], 1);
      mbar_init(&w_empty[s], 1 + 8 * NH);    // the products' commit, and every epilogue warp has read the biases
    }
    for (int b = 0; b < 2; ++b)
      for (int h = 0; h < 2; ++h) {
        mbar_init(&z_full[b][h], 1);
        mbar_init(&z_empty[b][h], 8);
      }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (threadIdx.x == 32) {
    prefetch_map(&maps.x);
    prefetch_map(&maps.hi);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;
  pdl_wait();
  pdl_trigger();

  const long long items = (long long)a.S * a.blocks;
  const long long it0 = first_item(items, a.n_cta, blockIdx.x), it1 = first_item(items, a.n_cta, blockIdx.x + 1);
  const int count = (int)(it1 - it0);
  const int g0 = (int)(it0 / a.blocks), b0 = (int)(it0 - (long long)g0 * a.blocks);

  if (warp == 0) {
    // ---------------------------------------------------------------- loads
    if (lane == 0) {
      bool ok = true;
      int g = g0, blk = b0, groups = 0, i = 0;
      for (; i < count; ++i) {
        if (i == 0 || blk == 0) {
          if (groups > 0) ok = mbar_wait(&grp_done, (groups - 1) & 1, abortp, a.status, 221);
          if (!ok) break;
          mbar_expect_tx(&x_full, kXBytes);
          tma_load_3d(x_s, &maps.x, &x_full, 0, 0, g);
          tma_load_3d(x_s + kXChunk, &maps.x, &x_full, 64, 0, g);
          ++groups;
        }
        const int s = i % kStages, n0 = blk * kLseCols;
        ok = mbar_wait(&w_empty[s], ((i / kStages) & 1) ^ 1, abortp, a.status, 222);
        if (!ok) break;
        const uint32_t bias_bytes = (uint32_t)min(kLseCols, a.ldw - n0) * 4;
        mbar_expect_tx(&w_full[s], kLseStage + bias_bytes);
        bulk_load(bias_s[s], a.bias + g * a.bias_sg + n0, bias_bytes, &w_full[s]);
        tma_load_3d(stages + s * kLseStage, &maps.hi, &w_full[s], n0, 0, g);
        tma_load_3d(stages + s * kLseStage + kTile, &maps.hi, &w_full[s], n0 + 64, 0, g);
        if (++blk == a.blocks) { blk = 0; ++g; }
      }
      if (!ok) {
        for (int j = max(0, i - kStages); j < i; ++j) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&w_full[j % kStages], (j / kStages) & 1) && clock64() - t0 < kWaitLimitCycles) {}
        }
        const long long t0 = clock64();
        while (groups > 0 && !mbar_try_wait(&x_full, (groups - 1) & 1) && clock64() - t0 < kWaitLimitCycles) {}
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- products
    const bool leader = elect_one();
    auto wait = [&](uint64_t* bar, uint32_t parity, int where) {
      return (bool)__all_sync(0xffffffffu, mbar_wait(bar, parity, abortp, a.status, where));
    };
    const int kz = (a.H + 15) / 16;
    const uint32_t id_z = make_idesc(0, 1, kLseCols, 128);
    const uint64_t x_k = make_desc(smem_u32(x_s), 16, 1024), w0 = make_desc(smem_u32(stages), kTile, 1024);
    bool ok = true;
    int blk = b0, groups = 0;
    bool fresh = true;
    for (int i = 0; i < count && ok; ++i) {
      if (fresh) ok = wait(&x_full, groups & 1, 223);
      const int s = i % kStages, b = i & 1;
      ok = ok && wait(&w_full[s], (i / kStages) & 1, 224);
      const uint64_t w = w0 + (uint64_t)((s * kLseStage) >> 4);
      for (int h = 0; h < NH && ok; ++h) {
        ok = wait(&z_empty[b][h], ((i >> 1) & 1) ^ 1, 225);
        if (!ok) break;
        tc_fence_after();
        const uint64_t x = x_k + (uint64_t)(h * 16384 >> 4);
        if (leader) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k < kz)
              tc_mma(tmem + b * 256 + h * 128, x + (((k >> 2) * kXChunk + (k & 3) * 32) >> 4), w + (k * 2048 >> 4), id_z, k != 0);
          tc_commit(&z_full[b][h]);
        }
        __syncwarp();
      }
      if (!ok) break;
      fresh = i + 1 == count || blk + 1 == a.blocks;
      if (leader) {
        tc_commit(&w_empty[s]);
        if (fresh) tc_commit(&grp_done);
      }
      __syncwarp();
      if (fresh) ++groups;
      if (++blk == a.blocks) blk = 0;
    }
  } else {
    // ---------------------------------------------------------------- sums of exponentials
    const int h = (warp - 2) >> 3, p = ((warp - 2) >> 2) & 1, q = warp & 3;
    const int row = h * 128 + q * 32 + lane;
    const uint32_t my_z = tmem + h * 128 + p * 64 + ((uint32_t)(q * 32) << 16);
    constexpr float kLog2e = 1.4426950408889634f;
    bool ok = h < NH;
    int g = g0, blk = b0;
    // sum of 2^(z log2e - ref) as sum + rest.  ref need not be the maximum, it only has to keep the sum inside the fp32
    // range: it stays where it is while a chunk's sum comes out moderate and moves to the chunk's maximum
    // otherwise (always for a thread's first chunk), so the common case has no comparison per element.
    float ref = -INFINITY, sum = 0.f, rest = 0.f;
    for (int i = 0; i < count && ok; ++i) {
      const int s = i % kStages, b = i & 1, n0 = blk * kLseCols + p * 64;
      ok = mbar_wait(&z_full[b][h], (i >> 1) & 1, abortp, a.status, 226) &&
           mbar_wait(&w_full[s], (i / kStages) & 1, abortp, a.status, 227);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const float* bias = bias_s[s] + p * 64;
      uint32_t both[64];
      tc_ld32(my_z + b * 256, both);
      tc_ld32(my_z + b * 256 + 32, both + 32);
      tc_fence_before();                     // z is in registers: the product of the block after the next may follow
      __syncwarp();
      if (lane == 0) mbar_arrive(&z_empty[b][h]);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const uint32_t* acc = both + 32 * c;
        float z[32];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float4 bv = *reinterpret_cast<const float4*>(bias + 32 * c + 4 * u);
          const float2 z0 = unpair(add2(pair(__uint_as_float(acc[4 * u + 0]), __uint_as_float(acc[4 * u + 1])), pair(bv.x, bv.y)));
          const float2 z1 = unpair(add2(pair(__uint_as_float(acc[4 * u + 2]), __uint_as_float(acc[4 * u + 3])), pair(bv.z, bv.w)));
          z[4 * u + 0] = z0.x; z[4 * u + 1] = z0.y; z[4 * u + 2] = z1.x; z[4 * u + 3] = z1.y;
        }
        const int nc = n0 + 32 * c;
        if (nc + 32 > a.N) {                 // the ragged end: columns beyond the classes do not count
          if (nc >= a.N) continue;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (nc + e >= a.N) z[e] = -INFINITY;
        }
        auto sum_exp = [&](float r) {        // four chains
          const f32x2 l2 = pair(kLog2e, kLog2e), nr = pair(-r, -r);
          f32x2 s0 = pair(0.f, 0.f), s1 = s0;
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float2 x0 = unpair(fma2(pair(z[e], z[e + 1]), l2, nr)), x1 = unpair(fma2(pair(z[e + 2], z[e + 3]), l2, nr));
            s0 = add2(s0, pair(ex2_approx(x0.x), ex2_approx(x0.y)));
            s1 = add2(s1, pair(ex2_approx(x1.x), ex2_approx(x1.y)));
          }
          const float2 t = unpair(add2(s0, s1));
          return t.x + t.y;
        };
        float cs = sum_exp(ref);
        // too large (2^64 or more; the exponent field also catches infinities and NaN), or below 2^-64 with nothing
        // to add it to: take the reference from this chunk
        const uint32_t cs_exp = (__float_as_uint(cs) >> 23) & 0xffu;
        if (cs_exp >= 127u + 64u || (cs_exp < 127u - 64u && sum == 0.f)) {
          float m4[4] = {z[0], z[1], z[2], z[3]};
#pragma unroll
          for (int e = 4; e < 32; ++e) m4[e & 3] = fmaxf(m4[e & 3], z[e]);
          const float mn = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * kLog2e;
          if (mn == -INFINITY) {             // a chunk of classes that biases rule out adds nothing, unless there is a NaN in it
            float any = 0.f;
#pragma unroll
            for (int e = 0; e < 32; ++e) any += z[e];
            cs = any != any ? any : 0.f;
          } else {
            if (sum != 0.f) {
              const float scale = ex2_approx(ref - mn);
              sum *= scale;
              rest *= scale;
            }
            ref = mn;
            cs = sum_exp(mn);
          }
        }
        const float t = sum + cs, bb = t - sum;   // what the addition rounds away is kept: hundreds of chunks follow one another
        rest += (sum - (t - bb)) + (cs - bb);
        sum = t;
        __syncwarp();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&w_empty[s]);
      if (i + 1 == count || blk + 1 == a.blocks) {
        const int part = (int)blockIdx.x - cta_of(items, a.n_cta, (long long)g * a.blocks);
        if (row < a.B) a.lse_part[((long long)g * a.partials + 2 * part + p) * a.B + row] = make_float2(ref, sum + rest);
        ref = -INFINITY;
        sum = rest = 0.f;
      }
      if (++blk == a.blocks) { blk = 0; ++g; }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// lse[g][b] from the rows' partials, a warp per row; the labels are checked here, as for every other output layer.
__global__ void __launch_bounds__(256) wide_lse_combine_kernel(const HeadArgs a, float* lse) {
  pdl_wait();
  pdl_trigger();
  const int rr = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (rr >= a.S * a.B) return;
  const int g = rr / a.B, row = rr - g * a.B;
  const long long items = (long long)a.S * a.blocks;
  const int parts = 2 * (cta_of(items, a.n_cta, (long long)(g + 1) * a.blocks - 1) - cta_of(items, a.n_cta, (long long)g * a.blocks) + 1);
  const float2* p = a.lse_part + (long long)g * a.partials * a.B + row;
  float m = -INFINITY;
  for (int i = lane; i < parts; i += 32) m = fmaxf(m, p[(long long)i * a.B].x);
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float s = 0.f;
  for (int i = lane; i < parts; i += 32) {
    const float2 v = p[(long long)i * a.B];
    if (v.y != 0.f) s += v.y * exp2f(v.x - m);   // a part of a ragged end may hold nothing
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    lse[g * a.lse_sg + row] = (m + log2f(s)) * 0.6931471805599453f;
    const int y = a.labels[g * a.labels_sg + row];
    if (y < 0 || y >= a.N) report(a.status, -5, SITE_LABEL, rr);
  }
}

// delta of the layer below: the subnet's dx partials added up in order, masked by that layer's activations; and the
// rows' losses.  One warp per row.
__global__ void __launch_bounds__(256) head_reduce_kernel(const HeadArgs a, const bf16* act, long long act_sg, bf16* out,
                                                          long long out_sg, float* row_loss) {
  pdl_wait();
  pdl_trigger();
  const int rr = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (rr >= a.S * a.B) return;
  const int g = rr / a.B, row = rr - g * a.B;
  const long long items = (long long)a.S * a.blocks;
  const int parts = cta_of(items, a.n_cta, (long long)(g + 1) * a.blocks - 1) - cta_of(items, a.n_cta, (long long)g * a.blocks) + 1;
  if (lane == 0) row_loss[rr] = a.lse[g * a.lse_sg + row] - a.label_logit[g * a.lse_sg + row];
  const int c = 4 * lane;
  if (c >= a.ldx) return;
  const float* p = a.dx_part + ((long long)g * a.partials * a.B + row) * a.ldx + c;
  const long long step = (long long)a.B * a.ldx;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int i = 0; i < parts; ++i) {
    float v[4];
    load4(p + i * step, v);
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] += v[e];
  }
  float m[4];
  load4(act + g * act_sg + (long long)row * a.ldx + c, m);
#pragma unroll
  for (int e = 0; e < 4; ++e) s[e] = m[e] > 0.f ? s[e] : 0.f;
  store4(out + g * out_sg + (long long)row * a.ldx + c, s);
}

int most_ctas(int S, int blocks, int n_cta) {   // that share a subnet
  const long long items = (long long)S * blocks;
  int most = 0;
  for (int g = 0; g < S; ++g)
    most = std::max(most, cta_of(items, n_cta, (long long)(g + 1) * blocks - 1) - cta_of(items, n_cta, (long long)g * blocks) + 1);
  return most;
}

// CTAs of the pass and dx partials per subnet; 0 CTAs: the scratch does not hold enough of them.
int plan_ctas(const WideHead& w, int sms, int* partials) {
  const int blocks = (int)ceil_div(w.N, kCols);
  const long long items = (long long)w.S * blocks;
  const long long cap = (long long)(w.scratch_bytes / ((size_t)w.S * w.B * w.ldx * 4));
  int n = (int)std::min<long long>(sms, items);
  for (;; --n) {
    if (n < 1) return 0;
    const int most = most_ctas(w.S, blocks, n);
    if (most <= cap) {
      *partials = most;
      return n;
    }
  }
}

}  // namespace

bool wide_head_ok(const WideHead& w) {
  int partials;
  return w.H <= 128 && w.ldx <= 128 && w.B <= 256 && plan_ctas(w, sm_count(), &partials) >= std::min<int64_t>(sm_count(), w.S * ceil_div(w.N, kCols)) / 2;
}

namespace {

// What both passes need; false: a tensor cannot be described to the copy engine.
bool common_args(const WideHead& w, int cols, DeviceStatus* st, HeadArgs* a, HeadMaps* m) {
  a->S = w.S; a->B = w.B; a->H = w.H; a->N = w.N; a->ldx = w.ldx; a->ldw = (int)w.ldw;
  a->blocks = (int)ceil_div(w.N, cols);
  a->halves = w.B > 128 ? 2 : 1;
  a->lr = w.lr; a->inv_rows = 1.f / (float)w.B;
  a->lse = w.lse; a->lse_sg = w.lse_sg; a->labels = w.labels; a->labels_sg = w.labels_sg; a->label_logit = w.label_logit;
  a->bias = w.bias; a->bias_sg = w.ldw;
  a->ties = w.ties;
  a->status = st;
  return make_map(&m->x, w.x, 2, w.H, w.B, w.S, w.ldx, w.x_sg, 64, 256, 128) &&
         make_map(&m->hi, w.opw, 2, w.N, w.H, w.S, w.ldw, w.w_sg, 64, 128, 128) &&
         make_map(&m->lo, w.lo, 2, w.N, w.H, w.S, w.ldw, w.w_sg, 64, 128, 128);
}

template <typename Kernel>
bool allow_smem(Kernel k, int bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
}

}  // namespace

bool wide_head_lse(const Launch& L, const WideHead& w, DeviceStatus* st) {
  HeadArgs a{};
  HeadMaps m;
  if (!common_args(w, kLseCols, st, &a, &m)) return false;
  a.n_cta = (int)std::min<int64_t>(sm_count(), (int64_t)w.S * a.blocks);
  a.partials = 2 * most_ctas(w.S, a.blocks, a.n_cta);
  a.lse_part = reinterpret_cast<float2*>(w.lse_part);
  static bool configured = false;
  static std::once_flag once;
  std::call_once(once, [] { configured = allow_smem(wide_lse_kernel, kLseSmem); });
  if (!configured) return false;
  if (launch_pdl(wide_lse_kernel, dim3(a.n_cta), dim3(kLseThreads), kLseSmem, L.stream, m, a) != cudaSuccess) return false;
  L.count();
  if (launch_pdl(wide_lse_combine_kernel, dim3((unsigned)ceil_div((int64_t)w.S * w.B, 8)), dim3(256), 0, L.stream, a, w.lse) !=
      cudaSuccess)
    return false;
  L.count();
  return true;
}

bool wide_head_pass(const Launch& L, const WideHead& w, DeviceStatus* st) {
  HeadArgs a{};
  HeadMaps m;
  a.n_cta = plan_ctas(w, sm_count(), &a.partials);
  if (a.n_cta < 1 || !common_args(w, kCols, st, &a, &m)) return false;
  a.dx_part = w.scratch;
  static bool configured = false;
  static std::once_flag once;
  std::call_once(once, [] { configured = allow_smem(wide_head_kernel, kSmem); });
  if (!configured) return false;
  if (launch_pdl(wide_head_kernel, dim3(a.n_cta), dim3(kThreads), kSmem, L.stream, m, a) != cudaSuccess) return false;
  L.count();
  if (launch_pdl(head_reduce_kernel, dim3((unsigned)ceil_div((int64_t)w.S * w.B, 8)), dim3(256), 0, L.stream, a, w.x, w.x_sg, w.delta,
                 w.x_sg, w.row_loss) != cudaSuccess)
    return false;
  L.count();
  return true;
}

}  // namespace ist
