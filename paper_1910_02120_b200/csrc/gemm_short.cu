// Grouped fp32 GEMM on the CUDA cores for short contractions (K <= 64): the small products of the
// fp32 path, where the tensor-core kernel's pipeline (gemm_f32.cu) would mostly be filling and draining.
//
// C[g](m, n) = sum_k A[g](m, k) * B[g](n, k) with arbitrary element strides: the same kernel serves
// x*W (B is n-contiguous), delta*W^T (B is k-contiguous) and a^T*delta (both operands contiguous
// along m / n).  A CTA computes a 32 x 32 tile, 2 x 2 per thread.  Such a launch is bound by latency
// alone, so the whole contraction is fetched at once: one round trip to memory, one barrier.
// Sums run over k in ascending order.
#include "bias_block.cuh"
#include "kernels.h"

namespace ist {
namespace {

constexpr int kThreads = 256, kTile = 32;

__device__ __forceinline__ void epilogue_store(const GemmArgs<float>& a, int g, int m, int n, float c) {
  switch (a.epi) {
    case EPI_BIAS_RELU:
      a.out[(int64_t)g * a.out_sg + (int64_t)m * a.out_ld + n] = fmaxf(c + a.bias[(int64_t)g * a.bias_sg + n], 0.f);
      break;
    case EPI_BIAS_F32:
      a.outf[(int64_t)g * a.outf_sg + (int64_t)m * a.outf_ld + n] = c + a.bias[(int64_t)g * a.bias_sg + n];
      break;
    case EPI_RELU_MASK: {
      const float mk = a.mask[(int64_t)g * a.mask_sg + (int64_t)m * a.mask_ld + n];
      a.out[(int64_t)g * a.out_sg + (int64_t)m * a.out_ld + n] = mk > 0.f ? c : 0.f;
      break;
    }
    case EPI_SGD: {
      float* w = a.outf + (int64_t)g * a.outf_sg + (int64_t)m * a.outf_ld + n;
      *w = *w - a.lr * c;
      break;
    }
    default:
      a.out[(int64_t)g * a.out_sg + (int64_t)m * a.out_ld + n] = c;
      break;
  }
}

struct ShortArgs {
  int n;
  GemmArgs<float> p[gemm_f32_max_batch()];
  int end[gemm_f32_max_batch()];            // blocks end(previous) .. end - 1 are the product's tiles
  BiasSgdArgs<float> bias;                  // blocks from end[n - 1] on, see bias_block
};

template <int KMAX>
__global__ void __launch_bounds__(kThreads) gemm_short_kernel(const __grid_constant__ ShortArgs args) {
  __shared__ float As[KMAX][kTile + 2];   // + 2: rows stay 8-byte aligned, transposing stores spread over the banks
  __shared__ float Bs[KMAX][kTile + 2];
  const int tid = threadIdx.x;
  if ((int)blockIdx.x >= args.end[args.n - 1]) {
    __shared__ float part[32][65];
    pdl_wait();
    pdl_trigger();
    bias_block(args.bias, blockIdx.x - args.end[args.n - 1], tid, part);
    return;
  }
  int pi = 0;
  while ((int)blockIdx.x >= args.end[pi]) ++pi;
  const GemmArgs<float>& a = args.p[pi];
  int tile = blockIdx.x - (pi ? args.end[pi - 1] : 0);
  const int n_tiles = (a.N + kTile - 1) / kTile, m_tiles = (a.M + kTile - 1) / kTile;
  const int n0 = tile % n_tiles * kTile;
  tile /= n_tiles;
  const int m0 = tile % m_tiles * kTile, g = tile / m_tiles;
  const float* A = a.A + (int64_t)g * a.a_sg;
  const float* B = a.B + (int64_t)g * a.b_sg;
  const bool a_k = a.a_sk == 1, b_k = a.b_sk == 1;   // consecutive lanes along k or along m / n
  constexpr int NE = kTile * KMAX / kThreads;
  float ra[NE], rb[NE];
  pdl_wait();
  pdl_trigger();
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = tid + kThreads * u;
    const int ka = a_k ? e % KMAX : e / kTile, ma = m0 + (a_k ? e / KMAX : e % kTile);
    const int kb = b_k ? e % KMAX : e / kTile, nb = n0 + (b_k ? e / KMAX : e % kTile);
    ra[u] = (ma < a.M && ka < a.K) ? A[(int64_t)ma * a.a_sm + (int64_t)ka * a.a_sk] : 0.f;
    rb[u] = (nb < a.N && kb < a.K) ? B[(int64_t)nb * a.b_sn + (int64_t)kb * a.b_sk] : 0.f;
  }
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = tid + kThreads * u;
    As[a_k ? e % KMAX : e / kTile][a_k ? e / KMAX : e % kTile] = ra[u];
    Bs[b_k ? e % KMAX : e / kTile][b_k ? e / KMAX : e % kTile] = rb[u];
  }
  __syncthreads();
  const int ty = tid / 16, tx = tid % 16;
  float c00 = 0.f, c01 = 0.f, c10 = 0.f, c11 = 0.f;
#pragma unroll 16
  for (int k = 0; k < a.K; ++k) {
    const float2 x = *reinterpret_cast<const float2*>(&As[k][2 * ty]);
    const float2 y = *reinterpret_cast<const float2*>(&Bs[k][2 * tx]);
    c00 = fmaf(x.x, y.x, c00); c01 = fmaf(x.x, y.y, c01);
    c10 = fmaf(x.y, y.x, c10); c11 = fmaf(x.y, y.y, c11);
  }
  const int m = m0 + 2 * ty, n = n0 + 2 * tx;
  if (m < a.M && n < a.N) epilogue_store(a, g, m, n, c00);
  if (m < a.M && n + 1 < a.N) epilogue_store(a, g, m, n + 1, c01);
  if (m + 1 < a.M && n < a.N) epilogue_store(a, g, m + 1, n, c10);
  if (m + 1 < a.M && n + 1 < a.N) epilogue_store(a, g, m + 1, n + 1, c11);
}

}  // namespace

bool gemm_short(const Launch& L, const GemmArgs<float>* a, int n, const BiasSgdArgs<float>* bias) {
  if (n < 1 || n > gemm_f32_max_batch()) return false;
  ShortArgs t{};
  t.n = n;
  int64_t end = 0;
  bool k32 = true;
  for (int i = 0; i < n; ++i) {
    if (a[i].M <= 0 || a[i].N <= 0 || a[i].G <= 0 || a[i].K > 64) return false;
    k32 &= a[i].K <= 32;
    end += ceil_div(a[i].N, kTile) * ceil_div(a[i].M, kTile) * a[i].G;
    if (end > 0x3fffffffll) return false;
    t.p[i] = a[i];
    t.end[i] = (int)end;
  }
  if (bias) {
    t.bias = *bias;
    end += bias_blocks(t.bias);
  }
  const dim3 grid((unsigned)end);
  const cudaError_t e = k32 ? launch_pdl(gemm_short_kernel<32>, grid, dim3(kThreads), 0, L.stream, t)
                            : launch_pdl(gemm_short_kernel<64>, grid, dim3(kThreads), 0, L.stream, t);
  if (e != cudaSuccess) return false;
  L.count();
  return true;
}

}  // namespace ist
