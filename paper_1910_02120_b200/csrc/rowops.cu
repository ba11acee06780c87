// Row-wise pieces of a local SGD step that are not contractions: softmax cross-entropy and
// its gradient, the bias update, input staging, and the evaluation reductions.
#include <algorithm>

#include "bias_block.cuh"
#include "kernels.h"

namespace ist {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide reductions with a fixed tree (deterministic for a given block size).
__device__ float block_max(float v, float* sh) {
  v = warp_max(v);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  float r = l < (blockDim.x >> 5) ? sh[l] : -INFINITY;
  return warp_max(r);
}
__device__ float block_sum(float v, float* sh) {
  v = warp_sum(v);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  float r = l < (blockDim.x >> 5) ? sh[l] : 0.f;
  return warp_sum(r);
}

// One CTA per row (g, b).  loss_row = log(sum exp(z - max)) + max - z[y];
// delta = (exp(z - max)/sum - [n == y]) / B.
template <typename T>
__global__ void softmax_xent_kernel(const float* logits, int64_t ld, int64_t sg, int B,
                                    int Nt, const int32_t* y, int64_t y_sg,
                                    T* __restrict__ delta, int64_t ld_d, int64_t sg_d,
                                    float* __restrict__ row_loss, DeviceStatus* st) {
  __shared__ float sh[32];
  pdl_wait();
  pdl_trigger();
  int g = blockIdx.y, b = blockIdx.x;
  const float* z = logits + (int64_t)g * sg + (int64_t)b * ld;
  T* d = delta + (int64_t)g * sg_d + (int64_t)b * ld_d;
  int label = y[(int64_t)g * y_sg + b];
  if (label < 0 || label >= Nt) {
    if (threadIdx.x == 0) report(st, -5, SITE_LABEL, (long long)g * B + b);
    label = 0;
  }
  float mx = -INFINITY;
  for (int n = threadIdx.x; n < Nt; n += blockDim.x) mx = fmaxf(mx, z[n]);
  mx = block_max(mx, sh);
  float se = 0.f;
  for (int n = threadIdx.x; n < Nt; n += blockDim.x) se += expf(z[n] - mx);
  se = block_sum(se, sh);
  float inv = 1.f / se, invB = 1.f / (float)B;
  for (int n = threadIdx.x; n < ld_d; n += blockDim.x) {
    float v = 0.f;
    if (n < Nt) v = (expf(z[n] - mx) * inv - (n == label ? 1.f : 0.f)) * invB;
    d[n] = from_float<T>(v);
  }
  if (threadIdx.x == 0) row_loss[(int64_t)g * B + b] = logf(se) + mx - z[label];
}

// Up to 32 V classes: one warp per row, eight rows per block, the row in registers.  The kernel above
// reads a row three times and crosses eight block barriers, all latency at these sizes (a local step of
// 256 rows of four subnets, 35 classes: 2 us less).  The exponentials are added in that kernel's order, so
// that a class count's results do not depend on which of the two takes it: row_threads(Nt) strided
// partial sums, a butterfly over each 32 of them, then the four warps' sums as (0 + 2) + (1 + 3).
template <typename T, int V>
__global__ void __launch_bounds__(256) softmax_xent_warp_kernel(const float* logits, int64_t ld, int64_t sg, int B,
                                                                int Nt, const int32_t* y, int64_t y_sg,
                                                                T* __restrict__ delta, int64_t ld_d, int64_t sg_d,
                                                                float* __restrict__ row_loss, DeviceStatus* st) {
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y, lane = threadIdx.x & 31, b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  const float* zr = logits + (int64_t)g * sg + (int64_t)b * ld;
  int label = y[(int64_t)g * y_sg + b];
  float z[V];
#pragma unroll
  for (int v = 0; v < V; ++v) z[v] = lane + 32 * v < Nt ? zr[lane + 32 * v] : -INFINITY;
  if (label < 0 || label >= Nt) {
    if (lane == 0) report(st, -5, SITE_LABEL, (long long)g * B + b);
    label = 0;
  }
  float mx = z[0];
#pragma unroll
  for (int v = 1; v < V; ++v) mx = fmaxf(mx, z[v]);
  mx = warp_max(mx);
  constexpr int W = V <= 2 ? 1 : 4;                    // warps of that block
  float part[W] = {}, zl = 0.f;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (lane + 32 * v == label) zl = z[v];
    z[v] = lane + 32 * v < Nt ? expf(z[v] - mx) : 0.f;
    part[v % W] += z[v];
  }
#pragma unroll
  for (int w = 0; w < W; ++w) part[w] = warp_sum(part[w]);
  const float se = W == 1 ? part[0] : (part[0] + part[2 % W]) + (part[1 % W] + part[3 % W]);
  zl = __shfl_sync(0xffffffffu, zl, label & 31);
  const float inv = 1.f / se, invB = 1.f / (float)B;
  T* d = delta + (int64_t)g * sg_d + (int64_t)b * ld_d;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int n = lane + 32 * v;
    if (n < ld_d) d[n] = from_float<T>(n < Nt ? (z[v] * inv - (n == label ? 1.f : 0.f)) * invB : 0.f);
  }
  if (lane == 0) row_loss[(int64_t)g * B + b] = logf(se) + mx - zl;
}

// Wide rows (hundreds of thousands of classes): one pass with a running (max, sum) pair per
// thread and 16-byte loads, then one pass that writes delta.  Row length ld is a multiple of 8.
template <typename T>
__global__ void __launch_bounds__(512) softmax_xent_wide_kernel(
    const float* logits, int64_t ld, int64_t sg, int B, int Nt, const int32_t* y,
    int64_t y_sg, T* __restrict__ delta, int64_t ld_d, int64_t sg_d, float* __restrict__ row_loss,
    DeviceStatus* st) {
  __shared__ float sm[16], ss[16];
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y, b = blockIdx.x;
  const float* z = logits + (int64_t)g * sg + (int64_t)b * ld;
  T* d = delta + (int64_t)g * sg_d + (int64_t)b * ld_d;
  int label = y[(int64_t)g * y_sg + b];
  if (label < 0 || label >= Nt) {
    if (threadIdx.x == 0) report(st, -5, SITE_LABEL, (long long)g * B + b);
    label = 0;
  }
  float m = -INFINITY, s = 0.f;
  const int nvec = Nt / 4;
  for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
    float4 t = *reinterpret_cast<const float4*>(z + 4 * v);
    float mx = fmaxf(fmaxf(t.x, t.y), fmaxf(t.z, t.w));
    if (mx > m) { s *= expf(m - mx); m = mx; }
    s += expf(t.x - m) + expf(t.y - m) + expf(t.z - m) + expf(t.w - m);
  }
  for (int n = nvec * 4 + threadIdx.x; n < Nt; n += blockDim.x) {
    float t = z[n];
    if (t > m) { s *= expf(m - t); m = t; }
    s += expf(t - m);
  }
  // combine (m, s) pairs: warp, then block
  for (int o = 16; o; o >>= 1) {
    float om = __shfl_xor_sync(0xffffffffu, m, o), os = __shfl_xor_sync(0xffffffffu, s, o);
    float nm = fmaxf(m, om);
    s = (m == -INFINITY ? 0.f : s * expf(m - nm)) + (om == -INFINITY ? 0.f : os * expf(om - nm));
    m = nm;
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sm[w] = m; ss[w] = s; }
  __syncthreads();
  float M = -INFINITY, S = 0.f;
  for (int u = 0; u < (int)(blockDim.x >> 5); ++u) {   // fixed order, every thread the same
    float nm = fmaxf(M, sm[u]);
    S = (M == -INFINITY ? 0.f : S * expf(M - nm)) + (sm[u] == -INFINITY ? 0.f : ss[u] * expf(sm[u] - nm));
    M = nm;
  }
  const float inv = 1.f / S, invB = 1.f / (float)B;
  const int nvec_d = (int)(ld_d / 4);
  for (int v = threadIdx.x; v < nvec_d; v += blockDim.x) {
    float o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int n = 4 * v + e;
      o[e] = n < Nt ? (expf(z[n] - M) * inv - (n == label ? 1.f : 0.f)) * invB : 0.f;
    }
    T* dst = d + 4 * v;
    dst[0] = from_float<T>(o[0]); dst[1] = from_float<T>(o[1]);
    dst[2] = from_float<T>(o[2]); dst[3] = from_float<T>(o[3]);
  }
  if (threadIdx.x == 0) row_loss[(int64_t)g * B + b] = logf(S) + M - z[label];
}

// Narrow output layer (Nt <= 64): one warp per row.  The logits may arrive as `ks` partial
// products of a k-split GEMM (slab g * ks + s holds slice s of group g, B rows of ld columns);
// they are summed here together with the bias, so the split costs no extra launch.
template <typename T>
__global__ void __launch_bounds__(256) softmax_xent_small_kernel(
    const float* part, int ks, int64_t ld, int B, int Nt, const float* bias,
    int64_t bias_sg, const int32_t* y, int64_t y_sg, T* __restrict__ delta, int64_t ld_d,
    int64_t sg_d, float* __restrict__ row_loss, DeviceStatus* st) {
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y, lane = threadIdx.x & 31;
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  int label = y[(int64_t)g * y_sg + b];
  if (label < 0 || label >= Nt) {
    if (lane == 0) report(st, -5, SITE_LABEL, (long long)g * B + b);
    label = 0;
  }
  // all slices are requested before the first is added (one after the other they were eight trips to L2)
  float z[2], slice[2][kHeadSplitsMax];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int n = lane + 32 * h;
    z[h] = n < Nt ? (bias ? bias[(int64_t)g * bias_sg + n] : 0.f) : -INFINITY;
#pragma unroll
    for (int s = 0; s < kHeadSplitsMax; ++s)
      slice[h][s] = (n < Nt && s < ks) ? part[(((int64_t)g * ks + s) * B + b) * ld + n] : 0.f;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int s = 0; s < kHeadSplitsMax; ++s)
      if (s < ks) z[h] += slice[h][s];   // fixed order
  const float mx = warp_max(fmaxf(z[0], z[1]));
  const float e0 = z[0] == -INFINITY ? 0.f : expf(z[0] - mx), e1 = z[1] == -INFINITY ? 0.f : expf(z[1] - mx);
  const float se = warp_sum(e0 + e1);
  const float zl = warp_sum((lane == (label & 31)) ? z[label >> 5] : 0.f);
  const float inv = 1.f / se, invB = 1.f / (float)B;
  T* d = delta + (int64_t)g * sg_d + (int64_t)b * ld_d;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int n = lane + 32 * h;
    if (n < ld_d) {
      const float e = h ? e1 : e0;
      d[n] = from_float<T>(n < Nt ? (e * inv - (n == label ? 1.f : 0.f)) * invB : 0.f);
    }
  }
  if (lane == 0) row_loss[(int64_t)g * B + b] = logf(se) + mx - zl;
}

// Bias gradient and update of every layer in one launch, blocks as bias_block wants them.
template <typename T>
__global__ void __launch_bounds__(256) bias_sgd_kernel(BiasSgdArgs<T> a) {
  __shared__ float part[32][65];
  pdl_wait();
  pdl_trigger();
  bias_block(a, blockIdx.x, threadIdx.x, part);
}

// lse[g][b] = log sum_n exp(z[g][b][n]) from per-tile partials (m, s) = (max of z * log2(e),
// sum of 2^(z * log2(e) - m)).  Block: 32 rows x 32 partial lanes; partials of one index are
// contiguous over rows.
__global__ void __launch_bounds__(1024) lse_combine_kernel(const float2* part, int parts, int B,
                                                            int64_t lse_sg, float* __restrict__ lse,
                                                            const int32_t* y, int64_t y_sg, int Nt,
                                                            DeviceStatus* st) {
  __shared__ float sm[32][33], ss[32][33];
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int b = blockIdx.x * 32 + tx;
  float m = -INFINITY, s = 0.f;
  if (b < B) {
    const float2* p = part + (int64_t)g * parts * B + b;
    // eight partials are requested before the first is folded in: a very wide layer has ten
    // thousand of them per row and only a few dozen blocks to read them
    constexpr int kAhead = 8;
    for (int i0 = ty; i0 < parts; i0 += 32 * kAhead) {
      float2 v[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int i = i0 + 32 * u;
        v[u] = i < parts ? p[(int64_t)i * B] : make_float2(-INFINITY, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        if (v[u].x > -INFINITY) {                  // an empty partial carries (-inf, 0)
          const float mn = fmaxf(m, v[u].x);
          s = s * exp2f(m - mn) + v[u].y * exp2f(v[u].x - mn);
          m = mn;
        }
      }
    }
  }
  sm[ty][tx] = m;
  ss[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && b < B) {
    float M = -INFINITY;
    for (int u = 0; u < 32; ++u) M = fmaxf(M, sm[u][tx]);
    float S = 0.f;
    for (int u = 0; u < 32; ++u)
      if (sm[u][tx] > -INFINITY) S += ss[u][tx] * exp2f(sm[u][tx] - M);
    lse[(int64_t)g * lse_sg + b] = (M + log2f(S)) * 0.6931471805599453f;
    const int label = y[(int64_t)g * y_sg + b];
    if (label < 0 || label >= Nt) report(st, -5, SITE_LABEL, (long long)g * B + b);
  }
}

__global__ void lse_row_loss_kernel(const float* lse, const float* zy, int B, int64_t lse_sg,
                                    float* __restrict__ row_loss) {
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y, b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) row_loss[(int64_t)g * B + b] = lse[(int64_t)g * lse_sg + b] - zy[(int64_t)g * lse_sg + b];
}

// A thread rounds four pairs of adjacent columns, their eight 4-byte loads (rows start at any 4-byte boundary)
// in flight together.  One block per row, or several (blockIdx.z) where the rows alone are too few to
// fill the GPU.  With a thread per element 1200 rows of 1001 took 10.7 us, now 6.7.
template <typename T>
__global__ void __launch_bounds__(128) stage_rows_kernel(const float* X, int64_t N0, int64_t group_row_stride,
                                                         T* __restrict__ out, int64_t ld, int64_t sg) {
  struct alignas(2 * sizeof(T)) Pair { T a, b; };
  constexpr int U = 4;
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x, g = blockIdx.y;
  const float* x = X + ((int64_t)g * group_row_stride + b) * N0;
  Pair* o = reinterpret_cast<Pair*>(out + (int64_t)g * sg + (int64_t)b * ld);   // ld is even, rows of `out` 16-byte aligned
  for (int64_t p0 = blockIdx.z * (U * 128) + threadIdx.x; p0 < ld / 2; p0 += gridDim.z * (U * 128)) {
    float v[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t c = 2 * (p0 + u * 128);
      v[u][0] = c < N0 ? x[c] : 0.f;
      v[u][1] = c + 1 < N0 ? x[c + 1] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (p0 + u * 128 < ld / 2) o[p0 + u * 128] = Pair{from_float<T>(v[u][0]), from_float<T>(v[u][1])};
  }
}

__global__ void eval_rows_kernel(const float* __restrict__ logits, int64_t ld, int rows, int Nt,
                                 const int32_t* __restrict__ y, double* loss_sum, long long* correct,
                                 DeviceStatus* st) {
  __shared__ float sh[32];
  __shared__ int shi[32];
  int r = blockIdx.x;
  const float* z = logits + (int64_t)r * ld;
  int label = y[r];
  if (label < 0 || label >= Nt) {
    if (threadIdx.x == 0) report(st, -5, SITE_LABEL, r);
    label = 0;
  }
  float mx = -INFINITY;
  int arg = 0x7fffffff;
  for (int n = threadIdx.x; n < Nt; n += blockDim.x) {
    float v = z[n];
    if (v > mx) { mx = v; arg = n; }   // first maximum inside the thread's strided set
  }
  // arg-max with lowest index on ties
  for (int o = 16; o; o >>= 1) {
    float om = __shfl_xor_sync(0xffffffffu, mx, o);
    int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (om > mx || (om == mx && oa < arg)) { mx = om; arg = oa; }
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sh[w] = mx; shi[w] = arg; }
  __syncthreads();
  if (w == 0) {
    float m2 = l < (blockDim.x >> 5) ? sh[l] : -INFINITY;
    int a2 = l < (blockDim.x >> 5) ? shi[l] : 0x7fffffff;
    for (int o = 16; o; o >>= 1) {
      float om = __shfl_xor_sync(0xffffffffu, m2, o);
      int oa = __shfl_xor_sync(0xffffffffu, a2, o);
      if (om > m2 || (om == m2 && oa < a2)) { m2 = om; a2 = oa; }
    }
    if (l == 0) { sh[0] = m2; shi[0] = a2; }
  }
  __syncthreads();
  mx = sh[0];
  arg = shi[0];
  float se = 0.f;
  for (int n = threadIdx.x; n < Nt; n += blockDim.x) se += expf(z[n] - mx);
  se = block_sum(se, sh);
  if (threadIdx.x == 0) {
    atomicAdd(loss_sum, (double)(logf(se) + mx - z[label]));
    if (arg == label) atomicAdd((unsigned long long*)correct, 1ull);
  }
}

// The same for rows of many classes: a cluster of CTAs per row, each with a range of the columns, one
// pass with a running (max, sum) pair and 16-byte loads, four of them in flight per thread; the
// ranges are merged in rank order through distributed shared memory.  Two passes of 4-byte loads by
// one block per row held too few bytes in flight for the 2.7 MB rows of 670,091 classes (256 rows:
// 2.46 ms; now 0.21 ms).
constexpr int kEvalThreads = 512, kEvalCols = 65536;   // a row is cut until a CTA has no more columns, or by eight
struct EvalPart { float m, s; int arg; };
// Folds b into a; ties go to the lower index.  An empty part carries (-inf, 0).
__device__ __forceinline__ void eval_fold(EvalPart& a, const EvalPart& b) {
  const float m = fmaxf(a.m, b.m), ref = m == -INFINITY ? 0.f : m;
  a.s = a.s * expf(a.m - ref) + b.s * expf(b.m - ref);
  if (b.m > a.m || (b.m == a.m && b.arg < a.arg)) a.arg = b.arg;
  a.m = m;
}
__global__ void __launch_bounds__(kEvalThreads) eval_rows_wide_kernel(const float* logits, int64_t ld, int Nt,
                                                                      const int32_t* y, double* loss_sum,
                                                                      long long* correct, DeviceStatus* st) {
  __shared__ EvalPart sh[kEvalThreads / 32];
  pdl_wait();
  pdl_trigger();
  const int row = blockIdx.y, rank = blockIdx.x, ranks = gridDim.x, tid = threadIdx.x;
  const float* z = logits + (int64_t)row * ld;
  const int per = (int)(((int64_t)Nt + ranks - 1) / ranks);
  const int c0 = min(rank * per, Nt), c1 = min(c0 + per, Nt);
  EvalPart p{-INFINITY, 0.f, 0x7fffffff};
  auto take = [&](const float* v, const int* at, int cnt) {
    float m = p.m;
#pragma unroll
    for (int i = 0; i < cnt; ++i)
      if (v[i] > m) { m = v[i]; p.arg = at[i]; }
    const float ref = m == -INFINITY ? 0.f : m;
    if (m > p.m) p.s *= expf(p.m - ref);
    p.m = m;
#pragma unroll
    for (int i = 0; i < cnt; ++i) p.s += expf(v[i] - ref);
  };
  // columns before the first 16-byte boundary and behind the last one by themselves
  const int head = min((int)((4 - ((reinterpret_cast<uintptr_t>(z + c0) >> 2) & 3)) & 3), c1 - c0);
  const int quads = (c1 - c0 - head) / 4;
  if (tid < head) { const int n = c0 + tid; take(z + n, &n, 1); }
  const float4* zq = reinterpret_cast<const float4*>(z + c0 + head);
  for (int q0 = tid; q0 < quads; q0 += 4 * kEvalThreads) {
    float v[16];
    int at[16];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = q0 + u * kEvalThreads;
      const float4 t = q < quads ? zq[q] : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      v[4 * u] = t.x; v[4 * u + 1] = t.y; v[4 * u + 2] = t.z; v[4 * u + 3] = t.w;
#pragma unroll
      for (int i = 0; i < 4; ++i) at[4 * u + i] = c0 + head + 4 * q + i;
    }
    take(v, at, 16);
  }
  const int tail = c0 + head + 4 * quads + tid;
  if (tail < c1) take(z + tail, &tail, 1);
  for (int o = 16; o; o >>= 1) {
    EvalPart q{__shfl_xor_sync(0xffffffffu, p.m, o), __shfl_xor_sync(0xffffffffu, p.s, o), __shfl_xor_sync(0xffffffffu, p.arg, o)};
    eval_fold(p, q);
  }
  if ((tid & 31) == 0) sh[tid >> 5] = p;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kEvalThreads / 32; ++w) eval_fold(p, sh[w]);
    sh[0] = p;
  }
  if (ranks > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (rank == 0 && tid == 0) {
    for (int r = 1; r < ranks; ++r) {
      uint32_t addr, w[3];
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"((uint32_t)__cvta_generic_to_shared(&sh[0])), "r"(r));
#pragma unroll
      for (int i = 0; i < 3; ++i) asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(w[i]) : "r"(addr + 4 * i) : "memory");
      eval_fold(p, EvalPart{__uint_as_float(w[0]), __uint_as_float(w[1]), (int)w[2]});
    }
    int label = y[row];
    if (label < 0 || label >= Nt) {
      report(st, -5, SITE_LABEL, row);
      label = 0;
    }
    atomicAdd(loss_sum, (double)(logf(p.s) + p.m - z[label]));
    if (p.arg == label) atomicAdd((unsigned long long*)correct, 1ull);
  }
  if (ranks > 1) {                                     // rank 0 has read the others' shared memory
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

__global__ void eval_finalize_kernel(const double* loss_sum, const long long* correct, int64_t n,
                                     float* mean_loss_out, int64_t* correct_out) {
  *mean_loss_out = (float)(*loss_sum / (double)n);
  *correct_out = (int64_t)*correct;
}

template <typename T>
__global__ void splitk_mask_reduce_kernel(const float* part, int ks, int B, int64_t ld,
                                          const T* mask, int64_t mask_sg, T* __restrict__ out,
                                          int64_t out_sg) {
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y;
  const int64_t per = (int64_t)B * ld;
  for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; e < per;
       e += (int64_t)gridDim.x * blockDim.x * 4) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < ks; ++s) {   // fixed order
      float4 v = *reinterpret_cast<const float4*>(part + ((int64_t)g * ks + s) * per + e);
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    const T* m = mask + (int64_t)g * mask_sg + e;
    T* o = out + (int64_t)g * out_sg + e;
    o[0] = from_float<T>(to_float(m[0]) > 0.f ? acc.x : 0.f);
    o[1] = from_float<T>(to_float(m[1]) > 0.f ? acc.y : 0.f);
    o[2] = from_float<T>(to_float(m[2]) > 0.f ? acc.z : 0.f);
    o[3] = from_float<T>(to_float(m[3]) > 0.f ? acc.w : 0.f);
  }
}

int row_threads(int Nt) { return Nt <= 64 ? 32 : (Nt <= 1024 ? 128 : kThreads); }

}  // namespace

template <typename T>
void softmax_xent(const Launch& L, const float* logits, int64_t ld, int64_t sg, int G, int B, int Nt,
                  const int32_t* y, int64_t y_sg, T* delta, int64_t ld_d, int64_t sg_d,
                  float* row_loss, DeviceStatus* st) {
  if (Nt > 8192 && ld % 4 == 0 && ld_d % 4 == 0)
    launch_pdl(softmax_xent_wide_kernel<T>, dim3(B, G), dim3(512), 0, L.stream, logits, ld, sg, B, Nt, y, y_sg, delta,
               ld_d, sg_d, row_loss, st);
  else if (Nt <= 1024) {   // a row fits the registers of a warp
    const dim3 grid((unsigned)ceil_div(B, 8), G);
    auto go = [&](auto kernel) {
      launch_pdl(kernel, grid, dim3(256), 0, L.stream, logits, ld, sg, B, Nt, y, y_sg, delta, ld_d, sg_d, row_loss, st);
    };
    if (Nt <= 64) go(softmax_xent_warp_kernel<T, 2>);
    else if (Nt <= 128) go(softmax_xent_warp_kernel<T, 4>);
    else if (Nt <= 512) go(softmax_xent_warp_kernel<T, 16>);
    else go(softmax_xent_warp_kernel<T, 32>);
  } else
    launch_pdl(softmax_xent_kernel<T>, dim3(B, G), dim3(row_threads(Nt)), 0, L.stream, logits, ld, sg, B, Nt, y, y_sg,
               delta, ld_d, sg_d, row_loss, st);
  L.count();
}
template void softmax_xent<float>(const Launch&, const float*, int64_t, int64_t, int, int, int,
                                  const int32_t*, int64_t, float*, int64_t, int64_t, float*,
                                  DeviceStatus*);
template void softmax_xent<bf16>(const Launch&, const float*, int64_t, int64_t, int, int, int,
                                 const int32_t*, int64_t, bf16*, int64_t, int64_t, float*,
                                 DeviceStatus*);

template <typename T>
void splitk_mask_reduce(const Launch& L, const float* part, int ks, int G, int B, int64_t ld, const T* mask,
                        int64_t mask_sg, T* out, int64_t out_sg) {
  const int64_t vecs = (int64_t)B * ld / 4;
  dim3 grid((unsigned)std::min<int64_t>(ceil_div(vecs, 256), 1024), G);
  launch_pdl(splitk_mask_reduce_kernel<T>, grid, dim3(256), 0, L.stream, part, ks, B, ld, mask, mask_sg, out, out_sg);
  L.count();
}
template void splitk_mask_reduce<bf16>(const Launch&, const float*, int, int, int, int64_t, const bf16*, int64_t,
                                       bf16*, int64_t);

template <typename T>
void softmax_xent_small(const Launch& L, const float* part, int ks, int64_t ld, int G, int B, int Nt,
                        const float* bias, int64_t bias_sg, const int32_t* y, int64_t y_sg, T* delta, int64_t ld_d,
                        int64_t sg_d, float* row_loss, DeviceStatus* st) {
  launch_pdl(softmax_xent_small_kernel<T>, dim3((unsigned)ceil_div(B, 8), G), dim3(256), 0, L.stream, part, ks, ld, B, Nt,
             bias, bias_sg, y, y_sg, delta, ld_d, sg_d, row_loss, st);
  L.count();
}
template void softmax_xent_small<bf16>(const Launch&, const float*, int, int64_t, int, int, int, const float*, int64_t,
                                       const int32_t*, int64_t, bf16*, int64_t, int64_t, float*, DeviceStatus*);

void lse_combine(const Launch& L, const float* lse_part, int parts, int G, int B, int64_t lse_sg, float* lse,
                 const int32_t* y, int64_t y_sg, int Nt, DeviceStatus* st) {
  launch_pdl(lse_combine_kernel, dim3((unsigned)ceil_div(B, 32), G), dim3(1024), 0, L.stream,
             reinterpret_cast<const float2*>(lse_part), parts, B, lse_sg, lse, y, y_sg, Nt, st);
  L.count();
}

void lse_row_loss(const Launch& L, const float* lse, const float* label_logit, int G, int B, int64_t lse_sg,
                  float* row_loss) {
  launch_pdl(lse_row_loss_kernel, dim3((unsigned)ceil_div(B, 256), G), dim3(256), 0, L.stream, lse, label_logit, B,
             lse_sg, row_loss);
  L.count();
}

template <typename T>
int bias_blocks(BiasSgdArgs<T>& a) {
  a.xstart[0] = 0;
  for (int i = 0; i < a.n_layers; ++i) a.xstart[i + 1] = a.xstart[i] + (int)ceil_div(a.layer[i].ld, 64);
  return (a.xstart[a.n_layers] + (a.loss.loss_out ? 1 : 0)) * a.G;
}
template int bias_blocks<float>(BiasSgdArgs<float>&);
template int bias_blocks<bf16>(BiasSgdArgs<bf16>&);

template <typename T>
void bias_sgd(const Launch& L, const BiasSgdArgs<T>& a) {
  BiasSgdArgs<T> b = a;
  const int blocks = bias_blocks(b);
  launch_pdl(bias_sgd_kernel<T>, dim3((unsigned)blocks), dim3(256), 0, L.stream, b);
  L.count();
}
template void bias_sgd<float>(const Launch&, const BiasSgdArgs<float>&);
template void bias_sgd<bf16>(const Launch&, const BiasSgdArgs<bf16>&);

template <typename T>
void stage_rows(const Launch& L, const float* X, int64_t N0, int64_t group_row_stride, int G, int B,
                T* out, int64_t ld, int64_t sg) {
  // sixteen blocks fit on an SM, 2368 on the GPU; a block beyond that, or beyond a row's 1024-column pieces, has nothing to do
  const int64_t pieces = std::max<int64_t>(1, std::min(ceil_div(ld, 1024), 2368 / ((int64_t)B * G)));
  launch_pdl(stage_rows_kernel<T>, dim3((unsigned)B, (unsigned)G, (unsigned)pieces), dim3(128), 0, L.stream, X, N0,
             group_row_stride, out, ld, sg);
  L.count();
}
template void stage_rows<float>(const Launch&, const float*, int64_t, int64_t, int, int, float*,
                                int64_t, int64_t);
template void stage_rows<bf16>(const Launch&, const float*, int64_t, int64_t, int, int, bf16*,
                               int64_t, int64_t);

void eval_rows(const Launch& L, const float* logits, int64_t ld, int rows, int Nt, const int32_t* y,
               double* loss_sum, long long* correct, DeviceStatus* st) {
  // From 4096 columns on a block's threads have a handful of 16-byte loads each.  As many CTAs per
  // row as keep the SMs supplied with two blocks each, at most the eight of a portable cluster.
  if (Nt >= 4096 && rows <= 65535) {
    int ranks = 1;
    while (ranks < 8 && ((int64_t)Nt / ranks > kEvalCols || ((int64_t)rows * ranks < 296 && Nt / ranks >= 8192))) ranks *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ranks, (unsigned)rows);
    cfg.blockDim = dim3(kEvalThreads);
    cfg.stream = L.stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)ranks;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, eval_rows_wide_kernel, logits, ld, Nt, y, loss_sum, correct, st);
  } else {
    eval_rows_kernel<<<rows, row_threads(Nt), 0, L.stream>>>(logits, ld, rows, Nt, y, loss_sum, correct, st);
  }
  L.count();
}

void eval_finalize(const Launch& L, const double* loss_sum, const long long* correct, int64_t n,
                   float* mean_loss_out, int64_t* correct_out) {
  eval_finalize_kernel<<<1, 1, 0, L.stream>>>(loss_sum, correct, n, mean_loss_out, correct_out);
  L.count();
}

}  // namespace ist
