// Calibration helper for the weight-activation product metric (Section 5, Stage 1: "if using calibration data is
// allowed ... weight-activation-product"): the Euclidean norm of every input channel over a set of tokens,
//   c[k] = sqrt(sum_m x[m][k]^2),
// which sdq_decompose_metric takes as its per-channel weight.  Accumulated in fp64, so the result is correctly rounded to
// fp32 for all practical sizes.
//
// Bound by reading X once.  A warp takes 64 channels (two per lane, one 128-byte line per token) and every 64th token: the
// eight warps of a CTA and the eight CTAs of a cluster share the tokens of a block of 64 channels, which puts enough lines
// in flight (one thread per two channels walking all tokens: 307 us for 2048 x 11008; this form: 16 us, 12 with X in L2).  The partial
// sums are added in a fixed order -- tokens of a warp, warps, CTAs -- whatever the size, so the result is reproducible.
#include <cuda_bf16.h>

#include "sdq_internal.h"
#include "sdq_ptx.cuh"

namespace sdq {

constexpr int CN_WARPS = 8, CN_CLUSTER = 8, CN_CHANNELS = 64;

__global__ void __cluster_dims__(1, CN_CLUSTER, 1) __launch_bounds__(32 * CN_WARPS)
channel_norm_kernel(const __nv_bfloat16* __restrict__ X, int64_t M, int64_t K, int64_t ldx, float* __restrict__ c)
{
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = ptx::cluster_ctarank();
  const int64_t k = (int64_t)blockIdx.x * CN_CHANNELS + lane * 2;       // K is even
  __shared__ double part[CN_WARPS][CN_CHANNELS], total[CN_CHANNELS];
  double s0 = 0.0, s1 = 0.0;
  if (k < K) {
    const __nv_bfloat16* col = X + k;
    constexpr int STEP = CN_WARPS * CN_CLUSTER, U = 8;                  // tokens between two of a warp; loads in flight
    int64_t m = (int64_t)rank * CN_WARPS + warp;
    auto add = [&](uint32_t r) {
      const double a = (double)__uint_as_float(r << 16), b = (double)__uint_as_float(r & 0xFFFF0000u);
      s0 += a * a;
      s1 += b * b;
    };
    for (; m + (U - 1) * STEP < M; m += U * STEP) {
      uint32_t r[U];
#pragma unroll
      for (int u = 0; u < U; ++u) r[u] = __ldg(reinterpret_cast<const uint32_t*>(col + (m + u * STEP) * ldx));
#pragma unroll
      for (int u = 0; u < U; ++u) add(r[u]);
    }
    for (; m < M; m += STEP) add(__ldg(reinterpret_cast<const uint32_t*>(col + m * ldx)));
  }
  part[warp][2 * lane] = s0;
  part[warp][2 * lane + 1] = s1;
  __syncthreads();
  if (threadIdx.x < CN_CHANNELS) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < CN_WARPS; ++w) s += part[w][threadIdx.x];
    total[threadIdx.x] = s;
  }
  ptx::cluster_sync();
  const int64_t ch = (int64_t)blockIdx.x * CN_CHANNELS + threadIdx.x;
  if (rank == 0 && threadIdx.x < CN_CHANNELS && ch < K) {
    double s = 0.0;
#pragma unroll
    for (uint32_t q = 0; q < CN_CLUSTER; ++q) {
      double v;
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ptx::mapa_u32(ptx::smem_u32(&total[threadIdx.x]), q)) : "memory");
      s += v;
    }
    c[ch] = (float)sqrt(s);
  }
  ptx::cluster_sync();                                                  // nobody leaves while its sums may still be read
}

}  // namespace sdq

using namespace sdq;

extern "C" sdq_status_t sdq_channel_norm(const void* X, int64_t M, int64_t K, int64_t ldx, float* col_norm, void* stream)
{
  if (!X || !col_norm) return SDQ_ERR_INVALID_ARG;
  if (M <= 0 || K <= 0 || (K & 1) || ldx < K) return SDQ_ERR_SHAPE;
  if (((uintptr_t)X & 3) || (ldx & 1) || ((uintptr_t)col_norm & 3)) return SDQ_ERR_ALIGNMENT;
  const dim3 grid((unsigned)((K + CN_CHANNELS - 1) / CN_CHANNELS), CN_CLUSTER);
  channel_norm_kernel<<<grid, 32 * CN_WARPS, 0, (cudaStream_t)stream>>>((const __nv_bfloat16*)X, M, K, ldx, col_norm);
  return cudaGetLastError() == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}
