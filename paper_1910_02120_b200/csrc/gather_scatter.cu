// Partition-indexed gather / scatter of weight slices between the full network and the
// per-subnet packed buffers (paper Sec. 2.1 "Constructing Subnets": a subnet's weights are the
// entries whose row and column neurons it owns; "Training Subnets": the trained slices go back
// to the positions they came from).  Pure data movement:
// fp32 values are moved bit for bit; the bf16 operand copy is a rounding of the moved value.  Masters that are kept
// as operand and low half (join_master) are taken apart and joined on the way.
#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace ist {
namespace {

// Packed elements o and o + 1 of a slice (o even): stored and loaded in whichever form the masters are kept in.  Pairs,
// because a thread that loads 2-byte halves one by one has half the bytes in flight (scatter of
// 3072-16384-16384-10, S = 8: 518 -> 395 us; 400 with fp32 words).
// Returns whether there is a tie, whose bit keep_tie must write.  Few are: a thread does that behind all its stores, with
// values read again, so that it costs no registers.
__device__ __forceinline__ bool put2(float* master, bf16* opw, uint16_t* lo, int64_t o, float v0, float v1) {
  uint32_t h, l, ties;
  split2(v0, v1, &h, &l, &ties);
  if (lo) *reinterpret_cast<uint32_t*>(lo + o) = l;
  else *reinterpret_cast<float2*>(master + o) = make_float2(v0, v1);
  if (opw) *reinterpret_cast<uint32_t*>(opw + o) = h;
  return lo && ((l & 0xffffu) == 0x8000u || l >> 16 == 0x8000u);
}
__device__ __forceinline__ uint32_t* ties_of(float* master) { return reinterpret_cast<uint32_t*>(master); }   // see SliceJob::lo
__device__ __forceinline__ void keep_tie(float* master, const SliceMap& m, int64_t s, int64_t i, int64_t j, float v) {
  const uint32_t u = __float_as_uint(v);
  if ((u & 0xffffu) != 0x8000u) return;
  const TieBit t = tie_bit(m.rows_pad, m.ld, s, i, j);
  if (u & 0x10000u) atomicAnd(ties_of(master) + t.word, ~t.mask);
  else atomicOr(ties_of(master) + t.word, t.mask);
}
// Loading is two steps, the words as they lie and then the values, so that a kernel has all its loads in flight
// first: a branch on the form around every load keeps the compiler from that.
template <bool SPLIT>
__device__ __forceinline__ uint2 raw2(const float* master, const bf16* opw, const uint16_t* lo, int64_t o) {
  if (!SPLIT) return *reinterpret_cast<const uint2*>(master + o);
  return make_uint2(*reinterpret_cast<const uint32_t*>(opw + o), *reinterpret_cast<const uint32_t*>(lo + o));
}
template <bool SPLIT>
__device__ __forceinline__ float2 value2(uint2 p) {
  if (!SPLIT) return make_float2(__uint_as_float(p.x), __uint_as_float(p.y));
  return make_float2(join_master((uint16_t)p.x, (uint16_t)p.y), join_master((uint16_t)(p.x >> 16), (uint16_t)(p.y >> 16)));
}
// The same for one element, where the positions of neighbours are not known to be a pair.
__device__ __forceinline__ bool put(float* master, bf16* opw, uint16_t* lo, int64_t o, float v) {
  const uint16_t l = (uint16_t)__float_as_uint(v);
  if (lo) lo[o] = l;
  else master[o] = v;
  if (opw) opw[o] = __float2bfloat16_rn(v);
  return lo && l == 0x8000;
}
template <bool SPLIT>
__device__ __forceinline__ float get(const float* master, const bf16* opw, const uint16_t* lo, int64_t o) {
  return SPLIT ? join_master(reinterpret_cast<const uint16_t*>(opw)[o], lo[o]) : master[o];
}
// Element (s, i, j) of a split slice, whichever of two ties it is.
__device__ __forceinline__ float settle(float* master, const SliceMap& m, int64_t s, int64_t i, int64_t j, float v) {
  if (!may_be_tie(v)) return v;
  const TieBit t = tie_bit(m.rows_pad, m.ld, s, i, j);
  return ties_of(master)[t.word] & t.mask ? other_tie(v) : v;
}

constexpr int kThreads = 256;
constexpr int kRowsPerCta = 4;

// Several matrices and bias rows as blocks of one launch: block -> (job, subnet, 4 rows, 512 columns).
// A network of a few layers took two launches per layer in either direction, most of them shorter
// than the gap between them (64-512-512-10, S = 4: 38 us to gather, 37 us to scatter; now 8.5 us each).
constexpr int kMaxJobs = 8;
struct SliceJobs {
  int n;
  SliceJob job[kMaxJobs];
  int x_blocks[kMaxJobs], y_blocks[kMaxJobs];
  int end[kMaxJobs];                 // blocks end(previous) .. end - 1 are the job's
};

// Packed element (s, i, j), j = column block * 512 + 2 tid (and j + 1), i in a block of kRowsPerCta rows.
// Pad rows / columns (beyond the group's true size) are written as zeros so that padded
// neurons stay inert through the local steps.
// Two rows at a time: with the loads of all rows in flight before the first store, the stores of a large matrix
// come in bursts that DRAM takes worse (middle layer of 32768 x 32768, S = 8: 1100 -> 1390 us for four rows).
template <bool SPLIT>
__device__ __forceinline__ void scatter_rows(const SliceJob& J, int s, int64_t j, const int64_t* c, const int32_t* rows, int64_t i0,
                                             int64_t i1) {
  const int64_t ld = J.m.ld, full = J.m.full_cols;
  int64_t o0 = ((int64_t)s * J.m.rows_pad + i0) * ld + j;
  for (int64_t i = i0; i < i1; i += 2, o0 += 2 * ld) {
    const bool two = i + 1 < i1;
    const uint2 p0 = raw2<SPLIT>(J.master, J.opw, J.lo, o0), p1 = two ? raw2<SPLIT>(J.master, J.opw, J.lo, o0 + ld) : p0;
    float* w0 = J.W + (rows ? rows[i] : i) * full;
    float* w1 = J.W + (two ? (rows ? rows[i + 1] : i + 1) * full : 0);
    float2 f0 = value2<SPLIT>(p0), f1 = value2<SPLIT>(p1);
    // both rows' loads have been asked for before this branch, which is hardly ever taken
    if (SPLIT && (may_be_tie(f0.x) | may_be_tie(f0.y) | may_be_tie(f1.x) | may_be_tie(f1.y))) {
      f0 = make_float2(settle(J.master, J.m, s, i, j, f0.x), settle(J.master, J.m, s, i, j + 1, f0.y));
      if (two) f1 = make_float2(settle(J.master, J.m, s, i + 1, j, f1.x), settle(J.master, J.m, s, i + 1, j + 1, f1.y));
    }
    w0[c[0]] = f0.x;
    if (c[1] >= 0) w0[c[1]] = f0.y;
    if (two) {
      w1[c[0]] = f1.x;
      if (c[1] >= 0) w1[c[1]] = f1.y;
    }
  }
}

template <bool GATHER>
__global__ void __launch_bounds__(kThreads) move_kernel(const __grid_constant__ SliceJobs a) {
  constexpr int R = kRowsPerCta;
  pdl_wait();
  pdl_trigger();
  int ji = 0, blk = blockIdx.x;
  while (blk >= a.end[ji]) ++ji;
  const SliceJob& J = a.job[ji];
  const SliceMap& m = J.m;
  blk -= ji ? a.end[ji - 1] : 0;
  const int64_t j = ((int64_t)(blk % a.x_blocks[ji]) * kThreads + threadIdx.x) * 2;   // columns j and j + 1
  blk /= a.x_blocks[ji];
  const int yb = blk % a.y_blocks[ji], s = m.s_first + blk / a.y_blocks[ji];
  if (!GATHER && J.mean) {
    for (int64_t n = j; n < min(j + 2, m.full_cols); ++n) {
      const float old = J.W[n];
      float acc = 0.f;
      for (int g = 0; g < J.S; ++g) acc += J.master[(int64_t)g * m.ld + n] - old;
      J.W[n] = old + acc / (float)J.S;
    }
    return;
  }
  const int64_t ncols = m.col_idx ? (m.col_off[s + 1] - m.col_off[s]) : m.full_cols;
  const int64_t nrows = m.row_idx ? (m.row_off[s + 1] - m.row_off[s]) : m.full_rows;
  if (j >= (GATHER ? m.ld : ncols)) return;
  int64_t c[2] = {-1, -1};
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (j + e < ncols) c[e] = m.col_idx ? m.col_idx[m.col_off[s] + j + e] : j + e;
  const int64_t i0 = (int64_t)yb * R;
  const int64_t o0 = ((int64_t)s * m.rows_pad + i0) * m.ld + j;
  if (!GATHER) {
    const int64_t i1 = min(i0 + R, nrows);
    const int32_t* rows = m.row_idx ? m.row_idx + m.row_off[s] : nullptr;
    if (J.lo) scatter_rows<true>(J, s, j, c, rows, i0, i1);
    else scatter_rows<false>(J, s, j, c, rows, i0, i1);
    return;
  }
  float v[R][2];
  int64_t r[R];
  bool tie = false;
#pragma unroll
  for (int u = 0; u < R; ++u)
    r[u] = i0 + u < nrows ? (m.row_idx ? m.row_idx[m.row_off[s] + i0 + u] : i0 + u) * m.full_cols : -1;
#pragma unroll
  for (int u = 0; u < R; ++u)
#pragma unroll
    for (int e = 0; e < 2; ++e) v[u][e] = r[u] >= 0 && c[e] >= 0 ? J.W[r[u] + c[e]] : 0.f;
#pragma unroll
  for (int u = 0; u < R; ++u)
    if (i0 + u < m.rows_pad) tie |= put2(J.master, J.opw, J.lo, o0 + u * m.ld, v[u][0], v[u][1]);
  if (tie)
#pragma unroll 1
    for (int64_t i = i0; i < min(i0 + R, nrows); ++i) {
      const float* w = J.W + (m.row_idx ? m.row_idx[m.row_off[s] + i] : i) * m.full_cols;
      keep_tie(J.master, m, s, i, j, w[c[0]]);               // c[0] >= 0: padding holds no tie
      if (c[1] >= 0) keep_tie(J.master, m, s, i, j + 1, w[c[1]]);
    }
}

// ---- last layer: whole rows, picked by the previous hidden layer's partition --------------------
// W_t[G_{t-1}^s, :] keeps every column, so both sides are contiguous along a row and the kernel is a
// strided row copy.  Rows of the full matrix start at any 4-byte offset (N_t is arbitrary), hence
// scalar accesses there, consecutive lanes on consecutive columns; a warp takes spans of 64 columns, of which a lane
// has columns l and 32 + l on that side and the pair 2 l, 2 l + 1 on the packed side, exchanged by shuffles.  A
// thread keeps kRowU x kColU values in flight, which is what the copy needs to approach the DRAM rate.
constexpr int kRowU = 4, kColU = 4;

// (columns l, 32 + l) of a span <-> (columns 2 l, 2 l + 1)
__device__ __forceinline__ void to_pairs(float& a, float& b) {
  const int lane = threadIdx.x & 31, src = 2 * (lane & 15);
  const float a0 = __shfl_sync(0xffffffffu, a, src), a1 = __shfl_sync(0xffffffffu, a, src + 1);
  const float b0 = __shfl_sync(0xffffffffu, b, src), b1 = __shfl_sync(0xffffffffu, b, src + 1);
  a = lane < 16 ? a0 : b0;
  b = lane < 16 ? a1 : b1;
}
__device__ __forceinline__ void from_pairs(float& a, float& b) {
  const int lane = threadIdx.x & 31, src = lane >> 1;
  const float a0 = __shfl_sync(0xffffffffu, a, src), b0 = __shfl_sync(0xffffffffu, b, src);
  const float a1 = __shfl_sync(0xffffffffu, a, 16 + src), b1 = __shfl_sync(0xffffffffu, b, 16 + src);
  a = lane & 1 ? b0 : a0;
  b = lane & 1 ? b1 : a1;
}

template <bool GATHER, bool SPLIT>
__global__ void __launch_bounds__(kThreads) rows_kernel(float* W, SliceMap m, float* master, bf16* opw,
                                                         uint16_t* lo) {
  pdl_wait();
  pdl_trigger();
  const int s = m.s_first + blockIdx.z;
  const int nrows = m.row_off[s + 1] - m.row_off[s];
  const int32_t* rows = m.row_idx + m.row_off[s];
  const int lane = threadIdx.x & 31;
  // this warp's spans of 64 columns start at j0 + c * kThreads, c = 0, 2, ...
  const int64_t j0 = (int64_t)blockIdx.x * (kThreads * kColU) + (threadIdx.x >> 5) * 64;
  for (int64_t i0 = (int64_t)blockIdx.y * kRowU; i0 < (GATHER ? m.rows_pad : nrows); i0 += (int64_t)gridDim.y * kRowU) {
    float v[kRowU][kColU];
    int64_t src[kRowU];
    bool tie = false;
#pragma unroll
    for (int u = 0; u < kRowU; ++u) src[u] = (i0 + u < nrows) ? (int64_t)rows[i0 + u] * m.full_cols : -1;
    if (GATHER) {
#pragma unroll
      for (int u = 0; u < kRowU; ++u)
#pragma unroll
        for (int c = 0; c < kColU; ++c) {
          const int64_t j = j0 + (c & ~1) * kThreads + (c & 1) * 32 + lane;
          v[u][c] = (src[u] >= 0 && j < m.full_cols) ? W[src[u] + j] : 0.f;   // pad rows / columns are zeros
        }
#pragma unroll
      for (int u = 0; u < kRowU; ++u)
#pragma unroll
        for (int c = 0; c < kColU; c += 2) {
          const int64_t j = j0 + c * kThreads + 2 * lane;
          to_pairs(v[u][c], v[u][c + 1]);
          if (i0 + u < m.rows_pad && j < m.ld)
            tie |= put2(master, opw, lo, ((int64_t)s * m.rows_pad + i0 + u) * m.ld + j, v[u][c], v[u][c + 1]);
        }
      if (tie)
#pragma unroll 1
        for (int e = 0; e < kRowU * kColU; ++e) {
          const int64_t i = i0 + e / kColU, j = j0 + (e % kColU & ~1) * kThreads + 2 * lane + (e & 1);
          if (i < nrows && j < m.full_cols) keep_tie(master, m, s, i, j, W[(int64_t)rows[i] * m.full_cols + j]);
        }
      __syncwarp();
    } else {
      uint2 p[kRowU][kColU / 2];
#pragma unroll
      for (int u = 0; u < kRowU; ++u)
#pragma unroll
        for (int c = 0; c < kColU; c += 2) {
          const int64_t j = j0 + c * kThreads + 2 * lane;
          p[u][c / 2] = (src[u] >= 0 && j < m.full_cols)
                            ? raw2<SPLIT>(master, opw, lo, ((int64_t)s * m.rows_pad + i0 + u) * m.ld + j) : make_uint2(0, 0);
        }
#pragma unroll
      for (int u = 0; u < kRowU; ++u)
#pragma unroll
        for (int c = 0; c < kColU; c += 2) {
          const float2 f = value2<SPLIT>(p[u][c / 2]);
          v[u][c] = f.x;
          v[u][c + 1] = f.y;
          from_pairs(v[u][c], v[u][c + 1]);
        }
#pragma unroll
      for (int u = 0; u < kRowU; ++u)
#pragma unroll
        for (int c = 0; c < kColU; ++c) {
          const int64_t j = j0 + (c & ~1) * kThreads + (c & 1) * 32 + lane;
          tie |= SPLIT && may_be_tie(v[u][c]);
          if (src[u] >= 0 && j < m.full_cols) W[src[u] + j] = v[u][c];
        }
      // ties are looked at again, each by the lane that stored it
      if (tie)
#pragma unroll 1
        for (int e = 0; e < kRowU * kColU; ++e) {
          const int64_t i = i0 + e / kColU, j = j0 + (e % kColU & ~1) * kThreads + (e & 1) * 32 + lane;
          if (i >= nrows || j >= m.full_cols) continue;
          float* w = W + (int64_t)rows[i] * m.full_cols + j;
          *w = settle(master, m, s, i, j, *w);
        }
      __syncwarp();
    }
  }
}

bool rows_ok(const SliceMap& m) { return m.row_idx && !m.col_idx && m.full_cols >= 1024; }

template <bool GATHER>
void launch_rows(const Launch& L, float* W, const SliceMap& m, int S, float* master, bf16* opw, uint16_t* lo) {
  dim3 grid((unsigned)ceil_div(m.ld, kThreads * kColU), (unsigned)std::min<int64_t>(ceil_div(m.rows_pad, kRowU), 65535), S);
  launch_pdl(lo ? rows_kernel<GATHER, true> : rows_kernel<GATHER, false>, grid, dim3(kThreads), 0, L.stream, W, m, master, opw, lo);
  L.count();
}

// ---- first layer: a column permutation, staged through shared memory -------------------------
// W_1[:, G_1^s] keeps whole rows and permutes their columns.  A CTA stages kStageRows rows x
// kStageCols consecutive columns (coalesced float4 accesses on the full-matrix side); because
// indices ascend inside a group, those columns form one contiguous run [lo_s, hi_s) in every
// group's packed row, so the packed side is coalesced as well.  The permutation itself is a
// random-access read (gather) or write (scatter) in shared memory.
constexpr int kStageRows = 8;
constexpr int kStageCols = 2048;
constexpr int kMaxGroupsStaged = 64;

struct ColRuns {                 // per group moved (m.s_first + i): packed positions [lo, lo + cnt) fall in the chunk
  int lo[kMaxGroupsStaged];
  int pre[kMaxGroupsStaged + 1]; // prefix sums of cnt
};

// First packed position of group s whose column index is >= c.
__device__ __forceinline__ int lower_bound_idx(const int32_t* idx, int n, int c) {
  int lo = 0, hi = n;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (idx[mid] < c) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ void find_runs(const SliceMap& m, int S, int c0, int c1, ColRuns* runs) {
  if (threadIdx.x < S) {
    const int s = m.s_first + threadIdx.x;
    const int32_t* g = m.col_idx + m.col_off[s];
    const int n = m.col_off[s + 1] - m.col_off[s];
    const int lo = lower_bound_idx(g, n, c0);
    runs->lo[threadIdx.x] = lo;
    runs->pre[threadIdx.x + 1] = lower_bound_idx(g, n, c1) - lo;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    runs->pre[0] = 0;
    for (int s = 0; s < S; ++s) runs->pre[s + 1] += runs->pre[s];
  }
  __syncthreads();
}

// ---- bulk-copy helpers (one thread moves whole row segments asynchronously) -------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void bar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
               ::"l"(dst), "r"(smem_addr(src_smem)), "r"(bytes) : "memory");
}

constexpr int kPermThreads = 512;
constexpr long long kPermWaitCycles = 2000000000ll;   // ~1 s

// Persistent CTA: column chunk blockIdx.x, row blocks blockIdx.y, blockIdx.y + gridDim.y, ...
// The map from a packed position of the chunk to (column inside the chunk, offset in the packed
// buffer) depends on the chunk only, so it is built once and reused for every row block.
// Gather: row blocks arrive through double-buffered bulk copies (the next block loads while
// this one is permuted).  Scatter: packed values are read into the permuted tile, which leaves
// through bulk stores.  Requires full_cols % 4 == 0 (16-byte row segments).
template <bool GATHER, bool SPLIT>
__global__ void __launch_bounds__(kPermThreads, 1) permute_cols_kernel(float* W, SliceMap m, int S,
                                                                      float* master, bf16* opw, uint16_t* lo,
                                                                      DeviceStatus* st) {
  extern __shared__ __align__(128) unsigned char perm_smem[];
  float* tile = reinterpret_cast<float*>(perm_smem);                                  // [2][rows][cols]
  long long* map_off = reinterpret_cast<long long*>(tile + 2 * kStageRows * kStageCols);   // [cols]
  uint16_t* map_col = reinterpret_cast<uint16_t*>(map_off + kStageCols);                   // [cols]
  __shared__ ColRuns runs;
  __shared__ uint64_t full[2];
  const int c0 = blockIdx.x * kStageCols;
  const int c1 = min((int)m.full_cols, c0 + kStageCols);
  const int width = c1 - c0;
  const int64_t n_blocks = ceil_div(m.full_rows, kStageRows);
  if (threadIdx.x == 0) {
    bar_init(&full[0], 1);
    bar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  pdl_wait();
  pdl_trigger();
  find_runs(m, S, c0, c1, &runs);      // contains the barriers that publish the mbarrier init
  const int total = runs.pre[S];
  for (int e = threadIdx.x; e < total; e += kPermThreads) {
    int i = 0;
    while (e >= runs.pre[i + 1]) ++i;
    const int s = m.s_first + i;
    const int j = runs.lo[i] + (e - runs.pre[i]);
    map_col[e] = (uint16_t)(m.col_idx[m.col_off[s] + j] - c0);
    map_off[e] = (long long)s * m.rows_pad * m.ld + j;
  }
  __syncthreads();

  auto issue_load = [&](int64_t rb, int buf) {   // thread 0 only
    const int64_t k0 = rb * kStageRows;
    const int nrows = (int)min((long long)kStageRows, (long long)(m.full_rows - k0));
    bar_expect_tx(&full[buf], (uint32_t)(nrows * width * 4));
    for (int r = 0; r < nrows; ++r)
      bulk_load(tile + (buf * kStageRows + r) * kStageCols, W + (k0 + r) * m.full_cols + c0, (uint32_t)(width * 4),
                &full[buf]);
  };

  if (GATHER && threadIdx.x == 0 && blockIdx.y < n_blocks) issue_load(blockIdx.y, 0);
  int it = 0;
  for (int64_t rb = blockIdx.y; rb < n_blocks; rb += gridDim.y, ++it) {
    const int buf = it & 1;
    const int64_t k0 = rb * kStageRows;
    const int nrows = (int)min((long long)kStageRows, (long long)(m.full_rows - k0));
    float* t = tile + buf * kStageRows * kStageCols;
    bool tie = false;                        // among this thread's values: they are gone through once more
    if (GATHER) {
      // the other buffer was last read in the previous iteration, which ended with a barrier
      if (threadIdx.x == 0 && rb + gridDim.y < n_blocks) issue_load(rb + gridDim.y, buf ^ 1);
      bool ok = true;
      const long long t0 = clock64();
      while (!bar_try_wait(&full[buf], (it >> 1) & 1)) {
        if (clock64() - t0 > kPermWaitCycles) { ok = false; break; }
      }
      if (!__syncthreads_and(ok)) {
        if (threadIdx.x == 0) report(st, -6, SITE_TC_PIPE, 100);
        return;
      }
      for (int e = threadIdx.x; e < total; e += kPermThreads) {
        const int col = map_col[e];
        const long long o = map_off[e] + k0 * m.ld;
#pragma unroll
        for (int r = 0; r < kStageRows; ++r)
          if (r < nrows) tie |= put(master, opw, lo, o + (long long)r * m.ld, t[r * kStageCols + col]);
      }
      if (tie)
#pragma unroll 1
        for (int e = threadIdx.x; e < total; e += kPermThreads) {
          const int64_t e0 = map_off[e];                       // of row 0: slab and column
          for (int r = 0; r < nrows; ++r) {
            const float v = t[r * kStageCols + map_col[e]];
            if ((uint16_t)__float_as_uint(v) == 0x8000) keep_tie(master, m, e0 / (m.rows_pad * m.ld), k0 + r, e0 % m.ld, v);
          }
        }
      if (blockIdx.x == 0) {   // pad columns [|G^s|, ld) of these rows are zero
        for (int s = m.s_first; s < m.s_first + S; ++s) {
          const int cnt = m.col_off[s + 1] - m.col_off[s];
          const int npad = (int)m.ld - cnt;
          for (int e = threadIdx.x; e < npad * nrows; e += kPermThreads) {
            const long long o = ((long long)s * m.rows_pad + k0 + e / npad) * m.ld + cnt + e % npad;
            put(master, opw, lo, o, 0.f);
          }
        }
      }
      __syncthreads();
    } else {
      // this buffer's previous stores (two iterations ago) must have read it
      if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      __syncthreads();
      for (int e = threadIdx.x; e < total; e += 2 * kPermThreads) {   // two entries' rows in flight
        const bool two = e + kPermThreads < total;
        const int col = map_col[e], col2 = two ? map_col[e + kPermThreads] : 0;
        const long long o = map_off[e] + k0 * m.ld, o2 = two ? map_off[e + kPermThreads] + k0 * m.ld : o;
        float v[kStageRows], v2[kStageRows];
#pragma unroll
        for (int r = 0; r < kStageRows; ++r) {
          v[r] = r < nrows ? get<SPLIT>(master, opw, lo, o + (long long)r * m.ld) : 0.f;
          v2[r] = r < nrows ? get<SPLIT>(master, opw, lo, o2 + (long long)r * m.ld) : 0.f;
        }
#pragma unroll
        for (int r = 0; r < kStageRows; ++r) {
          tie |= SPLIT && (may_be_tie(v[r]) | may_be_tie(v2[r]));
          t[r * kStageCols + col] = v[r];
          if (two) t[r * kStageCols + col2] = v2[r];
        }
      }
      if (tie)
#pragma unroll 1
        for (int e = threadIdx.x; e < total; e += kPermThreads) {
          const int64_t e0 = map_off[e];
          for (int r = 0; r < nrows; ++r) {
            float* v = t + r * kStageCols + map_col[e];
            if (may_be_tie(*v)) *v = settle(master, m, e0 / (m.rows_pad * m.ld), k0 + r, e0 % m.ld, *v);
          }
        }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int r = 0; r < nrows; ++r)
          bulk_store(W + (k0 + r) * m.full_cols + c0, t + r * kStageCols, (uint32_t)(width * 4));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    }
  }
  if (!GATHER && threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

bool staged_ok(const SliceMap& m, int S) {
  return !m.row_idx && m.col_idx && m.full_rows >= kStageRows && S <= kMaxGroupsStaged &&
         m.full_cols >= 256 && m.full_cols % 4 == 0;
}

template <bool GATHER, bool SPLIT>
bool launch_permute_cols(const Launch& L, float* W, const SliceMap& m, int S, float* master, bf16* opw, uint16_t* lo,
                         DeviceStatus* st) {
  constexpr int smem = 2 * kStageRows * kStageCols * (int)sizeof(float) + kStageCols * 8 + kStageCols * 2;
  static std::once_flag once;     // one instance per direction; any host thread may come first
  static bool configured = false;
  std::call_once(once, [] {
    configured = cudaFuncSetAttribute(permute_cols_kernel<GATHER, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem) == cudaSuccess;
  });
  if (!configured) return false;
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t chunks = ceil_div(m.full_cols, kStageCols), blocks = ceil_div(m.full_rows, kStageRows);
  int64_t y = sms / chunks;
  if (y < 1) y = 1;
  if (y > blocks) y = blocks;
  if (y > 65535) y = 65535;
  dim3 grid((unsigned)chunks, (unsigned)y);
  if (launch_pdl(permute_cols_kernel<GATHER, SPLIT>, grid, dim3(kPermThreads), smem, L.stream, W, m, S, master, opw, lo, st) != cudaSuccess)
    return false;
  L.count();
  return true;
}

__global__ void copy_out_kernel(const SliceJob job, int s, int64_t rows, int64_t cols, float* __restrict__ out) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t i = blockIdx.y;
  if (j < cols)
    for (; i < rows; i += gridDim.y) {
      const int64_t o = ((int64_t)s * job.m.rows_pad + i) * job.m.ld + j;
      out[i * cols + j] = job.lo ? settle(job.master, job.m, s, i, j, get<true>(job.master, job.opw, job.lo, o)) : job.master[o];
    }
}

// Masters first .. end - 1 of n become fp32 words in place.  The low halves are the second half of the words, so
// word i takes the place of low halves 2 i - n and 2 i - n + 1, both at or before i: a launch may cover words as long as
// they replace only low halves of words before its first.  One block may end the array: it reads all it needs
// before it writes.  The first words replace the tie bits, so ties that rounded down get the operand that rounding up would
// give them before, which joins to their value, and their operands are put right here.
__global__ void write_out_ties_kernel(const SliceJob job, int64_t n) {
  uint16_t* hi = reinterpret_cast<uint16_t*>(job.opw);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (job.lo[i] != 0x8000 || (hi[i] & 1)) continue;
    const TieBit t = tie_bit(job.m.rows_pad, job.m.ld, i / (job.m.rows_pad * job.m.ld), i / job.m.ld % job.m.rows_pad, i % job.m.ld);
    if (ties_of(job.master)[t.word] & t.mask) hi[i] += 1;
  }
}
__device__ __forceinline__ void join_one(const SliceJob& job, int64_t i, float w) {
  const bf16 operand = __float2bfloat16_rn(w);
  if (__bfloat16_as_ushort(job.opw[i]) != __bfloat16_as_ushort(operand)) job.opw[i] = operand;
  job.master[i] = w;
}
__global__ void join_masters_kernel(const SliceJob job, int64_t first, int64_t end) {
  if (gridDim.x > 1) {
    for (int64_t i = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end; i += (int64_t)gridDim.x * blockDim.x)
      join_one(job, i, get<true>(job.master, job.opw, job.lo, i));
  } else {
    const int64_t i = first + threadIdx.x;
    const float w = i < end ? get<true>(job.master, job.opw, job.lo, i) : 0.f;
    __syncthreads();
    if (i < end) join_one(job, i, w);
  }
}

}  // namespace

namespace {

// Matrices of this many packed elements or more are moved by the kernel made for their kind (first
// layer: column permutation, last layer: whole rows); smaller ones by blocks of the shared launch,
// whose scattered 4-byte accesses L2 still absorbs.  Partition + reassembly with the large matrix in the shared
// launch and in one of its own, S = 1 / 16 subnets, bf16 operands, us:
//   first layer  1024 x 4096   51 / 62   against  55 / 59     last layer  3072 x 1024  44 / 44   against  38 / 39
//                1536 x 4096   58 / 77            59 / 66                 4096 x 1024  50 / 50            41 / 43
//                768 x 16384  114 / 144          111 / 121                8192 x 1024  75 / 75            50 / 53
//   3072 x 16384, S = 8: 1180 against 740                                 5003 x 3000 112 / 114           74 / 76
// The column permutation has a fixed part of some 10 us, which few subnets do not repay below 12 M.
constexpr int64_t kOwnColumns = 12 << 20, kOwnRows = 3 << 20;

template <bool GATHER>
void move_all(const Launch& L, const SliceJob* jobs, int n, DeviceStatus* st) {
  SliceJobs a{};
  int64_t blocks = 0;
  auto flush = [&] {
    if (a.n) {
      launch_pdl(move_kernel<GATHER>, dim3((unsigned)blocks), dim3(kThreads), 0, L.stream, a);
      L.count();
    }
    a.n = 0;
    blocks = 0;
  };
  for (int i = 0; i < n; ++i) {
    const SliceJob& j = jobs[i];
    const int64_t elements = j.mean ? 0 : j.S * j.m.rows_pad * j.m.ld;
    if (elements >= kOwnColumns && staged_ok(j.m, j.S)) {
      const auto launch = j.lo ? launch_permute_cols<GATHER, true> : launch_permute_cols<GATHER, false>;
      if (launch(L, j.W, j.m, j.S, j.master, j.opw, j.lo, st)) continue;
    }
    if (elements >= kOwnRows && rows_ok(j.m)) {
      launch_rows<GATHER>(L, j.W, j.m, j.S, j.master, j.opw, j.lo);
      continue;
    }
    const int64_t x = ceil_div(j.mean ? j.m.full_cols : j.m.ld, 2 * kThreads), y = j.mean ? 1 : ceil_div(j.m.rows_pad, kRowsPerCta);
    const int64_t b = x * y * (j.mean ? 1 : j.S);
    if (a.n == kMaxJobs || blocks + b > 0x7fffffffll) flush();
    a.job[a.n] = j;
    a.x_blocks[a.n] = (int)x;
    a.y_blocks[a.n] = (int)y;
    blocks += b;
    a.end[a.n++] = (int)blocks;
  }
  flush();
}

}  // namespace

void gather_slices(const Launch& L, const SliceJob* jobs, int n, DeviceStatus* st) { move_all<true>(L, jobs, n, st); }
void scatter_slices(const Launch& L, const SliceJob* jobs, int n, DeviceStatus* st) { move_all<false>(L, jobs, n, st); }

void copy_out_slice(const Launch& L, const SliceJob& j, int s, int64_t rows, int64_t cols, float* out) {
  dim3 grid((unsigned)ceil_div(cols, 256), (unsigned)(rows < 1024 ? rows : 1024));
  copy_out_kernel<<<grid, 256, 0, L.stream>>>(j, s, rows, cols, out);
  L.count();
}

void join_masters(const Launch& L, const SliceJob& j) {
  constexpr int kJoin = 1024;
  const int64_t n = j.S * j.m.rows_pad * j.m.ld;
  write_out_ties_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n, kJoin), 4096), kJoin, 0, L.stream>>>(j, n);
  L.count();
  int64_t first = 0;
  while (first < n) {
    int64_t end = first + (n - first) / 2;     // words below this replace low halves below `first` only
    if (n - first <= kJoin) end = n;
    const int64_t blocks = n - first <= kJoin ? 1 : std::max<int64_t>(2, std::min<int64_t>(ceil_div(end - first, kJoin), 4096));
    join_masters_kernel<<<(unsigned)blocks, kJoin, 0, L.stream>>>(j, first, end);
    L.count();
    first = end;
  }
}

}  // namespace ist
