// A narrow output layer on the fp32 path, from the activations below it to their delta: logits, softmax cross-entropy with
// its gradient, and delta_{t-1} = (delta_t W_t^T) masked by a_{t-1} > 0 (paper Sec. 2.1, the steps of one local update).
//
// What bounds it: latency; as three launches these were 3 to 4 us each for a few hundred thousand products.  A block takes
// eight rows, with the layer's weights and the rows in shared memory: one trip to L2 for all three, and two barriers
// between them instead of two launches.
// Per step of the whole chain: 64-256-256-10, S = 4, 64 rows 26.6 -> 21.3 us; 784-1024-10, S = 2, 128 rows 37.2 -> 31.5.
// Logits of up to 64 neurons are one chain of products in ascending order, bit for bit those of gemm_short_kernel; those of
// more are chains of 32, added up in four sums.  The exponentials are added like softmax_xent_warp_kernel's, delta_{t-1} is a
// chain over the classes.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "tma_map.h"

namespace ist {
namespace {

constexpr int kThreads = 256, kRows = 8, kMaxClasses = 64;
constexpr int kSmemLimit = 227 * 1024, kSmemPerSm = 228 * 1024;
constexpr int64_t kMaxWork = 26000;

struct HeadF32Args {
  HeadF32 h;
  int pa, pw;                              // row lengths of activations and weights in shared memory
  int chain, chunks;                       // products of a chain, chains per logit
  DeviceStatus* status;
};

__device__ __forceinline__ void copy16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float warp_total(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(kThreads) head_f32_kernel(const __grid_constant__ HeadF32Args args) {
  const HeadF32& h = args.h;
  extern __shared__ __align__(16) float sm[];
  const int K = h.H, N = h.N, pa = args.pa, pw = args.pw;
  float* a_s = sm;                               // [8][pa]
  float* w_s = a_s + kRows * pa;                 // [K rounded up to 4][pw]
  float* d_s = w_s + ((K + 3) & ~3) * pw;        // [8][64]: delta_t
  float* part = d_s + kRows * kMaxClasses;       // [chunks][8][N]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = blockIdx.y, m0 = blockIdx.x * kRows;
  // the last step of four products may reach past the neurons
  for (int i = tid; i < ((K + 3) & ~3) * pw - K * pw; i += kThreads) w_s[K * pw + i] = 0.f;
  pdl_wait();
  pdl_trigger();
  {
    const float* W = h.W + (long long)g * h.w_sg;
    const int quads = (int)(h.ldw >> 2);         // whole padded rows
    for (int i = tid; i < K * quads; i += kThreads) {
      const int r = i / quads, q = i - r * quads;
      copy16(w_s + r * pw + 4 * q, W + (long long)r * h.ldw + 4 * q);
    }
    const int m = min(m0 + warp, h.B - 1);       // a warp per row; rows behind the batch repeat its last
    const float* x = h.x + (long long)g * h.x_sg + (long long)m * h.ldx;
    for (int q = lane; q < (K + 3) >> 2; q += 32) copy16(a_s + warp * pa + 4 * q, x + 4 * q);
  }
  float bias[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) bias[v] = lane + 32 * v < N ? h.bias[(long long)g * h.ldw + lane + 32 * v] : 0.f;
  const int m = m0 + warp;
  int label = m < h.B ? h.labels[(long long)g * h.labels_sg + m] : 0;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  if (lane < ((K + 3) & ~3) - K) a_s[warp * pa + K + lane] = 0.f;
  __syncthreads();

  // ---- chains of the logits: class, then four rows, then chain
  for (int it = tid; it < args.chunks * 2 * N; it += kThreads) {
    const int q = it / N, n = it - q * N, r0 = (q & 1) * 4, k0 = (q >> 1) * args.chain, k1 = min(K, k0 + args.chain);
    const float* a = a_s + r0 * pa;
    const float* w = w_s + n;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int k = k0; k < k1; k += 4) {
      const float u[4] = {w[k * pw], w[(k + 1) * pw], w[(k + 2) * pw], w[(k + 3) * pw]};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(a + i * pa + k);
        c[i] = fmaf(x.w, u[3], fmaf(x.z, u[2], fmaf(x.y, u[1], fmaf(x.x, u[0], c[i]))));
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) part[((q >> 1) * kRows + r0 + i) * N + n] = c[i];
  }
  __syncthreads();

  // ---- a warp per row: softmax, delta_t, the row's loss
  {
    float z[2], e[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int n = lane + 32 * v;
      z[v] = -INFINITY;
      if (n < N) {
        float s[4] = {part[warp * N + n], 0.f, 0.f, 0.f};
        for (int c = 1; c < args.chunks; c += 4)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (c + u < args.chunks) s[u] += part[((c + u) * kRows + warp) * N + n];
        z[v] = ((s[0] + s[1]) + (s[2] + s[3])) + bias[v];
      }
    }
    if (label < 0 || label >= N) {
      if (lane == 0) report(args.status, -5, SITE_LABEL, (long long)g * h.B + m);
      label = 0;
    }
    float mx = fmaxf(z[0], z[1]), zl = 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      if (lane + 32 * v == label) zl = z[v];
      e[v] = lane + 32 * v < N ? expf(z[v] - mx) : 0.f;
    }
    const float se = warp_total(e[0] + e[1]);
    zl = __shfl_sync(0xffffffffu, zl, label & 31);
    const float inv = 1.f / se, inv_rows = 1.f / (float)h.B;
    float* d = h.delta_out + (long long)g * h.dout_sg + (long long)m * h.ldw;
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int n = lane + 32 * v;
      const float o = n < N ? (e[v] * inv - (n == label ? 1.f : 0.f)) * inv_rows : 0.f;
      d_s[warp * kMaxClasses + n] = o;
      if (m < h.B && n < h.ldw) d[n] = o;
    }
    if (lane == 0 && m < h.B) h.row_loss[(long long)g * h.B + m] = logf(se) + mx - zl;
  }
  __syncthreads();

  // ---- delta of the layer below, a thread per neuron
  for (int k = tid; k < K; k += kThreads) {
    const float* w = w_s + k * pw;
    float c[kRows] = {};
    int n = 0;
    for (; n + 4 <= N; n += 4) {
      const float4 u = *reinterpret_cast<const float4*>(w + n);
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(d_s + r * kMaxClasses + n);
        c[r] = fmaf(x.w, u.w, fmaf(x.z, u.z, fmaf(x.y, u.y, fmaf(x.x, u.x, c[r]))));
      }
    }
    for (; n < N; ++n)
#pragma unroll
      for (int r = 0; r < kRows; ++r) c[r] = fmaf(d_s[r * kMaxClasses + n], w[n], c[r]);
#pragma unroll
    for (int r = 0; r < kRows; ++r)
      if (m0 + r < h.B)
        h.delta[(long long)g * h.x_sg + (long long)(m0 + r) * h.ldx + k] = a_s[r * pa + k] > 0.f ? c[r] : 0.f;
  }
}

// Bytes of shared memory of a block.
int64_t lay_out(const HeadF32& h, HeadF32Args* a) {
  const int64_t k4 = round_up(h.H, 4);
  a->pa = (int)k4 + 4;                           // + 4: consecutive rows' 16-byte units lie in different banks
  a->pw = (int)h.ldw + 4;
  a->chain = h.H <= 64 ? 64 : 32;
  a->chunks = (int)ceil_div(h.H, a->chain);
  return 4 * (kRows * (k4 + 4) + k4 * (h.ldw + 4) + kRows * kMaxClasses + (int64_t)a->chunks * kRows * h.N);
}

}  // namespace

// A block's time goes with the layer's weights, and blocks follow one another in rounds.  Up to 26,000 weights times rounds no
// step measured slower than with three launches: 400 x 64 with 24 rows 22.1 us either way, with 4 x 256 rows 38.8 -> 35.2,
// 250 x 40 with 8 x 640 rows (two rounds) 57.1 -> 50.4, 256 x 10 with 16 x 640 78.3 -> 57.9; beyond, 512 x 64 with 2 x 16 rows
// took 23.9 for 21.2 and 500 x 64 with 2 x 640 (two rounds) 48.5 for 38.4.
bool head_f32_ok(const HeadF32& h) {
  HeadF32Args a{};
  if (h.N > kMaxClasses || h.H > 16384) return false;
  const int64_t bytes = lay_out(h, &a);
  if (bytes > kSmemLimit) return false;
  const int64_t resident = std::min<int64_t>(8, kSmemPerSm / (bytes + 1024));
  const int64_t rounds = ceil_div(ceil_div(h.B, kRows) * h.S, resident * sm_count());
  return rounds * h.H * h.N <= kMaxWork;
}

bool head_f32(const Launch& L, const HeadF32& h, DeviceStatus* st) {
  HeadF32Args a{};
  const int64_t bytes = lay_out(h, &a);
  a.h = h;
  a.status = st;
  static bool configured = false;
  static std::once_flag once;
  std::call_once(once, [] {
    configured = cudaFuncSetAttribute(head_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) == cudaSuccess;
  });
  if (!configured) return false;
  if (launch_pdl(head_f32_kernel, dim3((unsigned)ceil_div(h.B, kRows), (unsigned)h.S), dim3(kThreads), (size_t)bytes, L.stream, a) !=
      cudaSuccess)
    return false;
  L.count();
  return true;
}

}  // namespace ist
