// fp32 contraction with whole rows in shared memory, the RMSNorm of its input folded in.
//
//   C[t, f] (op)= sum_k A'[t, k] * W[f, k]       A' = A, or gain * A / sqrt(mean(A^2) + eps)
//
// The fp32 models are small (rows of 64 ... 512 features), so a contraction is a link of a chain of
// dependent launches and costs what its memory round trips cost.  The 64 x 64 tile of
// gemm_simt_kernel makes one such round trip per 16 features of K; here a CTA requests its weight
// rows before the dependency wait and its whole activation rows in one go behind it, and since it
// holds the rows it also normalises them: the RMSNorm launch in front of the contraction goes away.
//   * tile MT tokens x FN features over the whole K; the eight warps take the 4-feature vectors of K
//     in turn (vector w, w + 8, ...), each lane accumulating (MT / 4) x (FN / 8) outputs in fp32 FMAs;
//     the partial tiles are summed through shared memory in warp order, so every epilogue sees
//     complete sums and the order of the additions is fixed;
//   * rows are padded by 16 bytes: the four token rows and eight feature rows that a warp reads at a
//     time fall into different banks.
// Bound: latency (launch, one L2 round trip, the 8-way sum); 3.5 us a link inside a captured forecast where
// the 64 x 64 tile took 8 to 31 us (M = 37 ... 185, K = 128, 512).  Forecast of one series with the 2-layer
// d = 128 model: 636 -> 260 us; of 37 series 2.55 -> 0.90 ms.
// grid = (ceil(N / FN), ceil(M / MT)), block = 256.  K a multiple of 16.
#pragma once
#include "common.cuh"
#include "kernels_simt.cuh"

namespace tsfm {

template <int MT, int FN> constexpr int f32_smem_bytes(int K) {
  const int rows = (MT + FN) * (K + 4) * 4, red = 8 * MT * FN * 4;      // the partial sums reuse the rows
  return rows > red ? rows : red;
}

template <int MT, int FN>
__global__ void __launch_bounds__(256)
gemm_f32_kernel(const float *A, const float *__restrict__ W, float *C, int M, int N, int K, int epi,
                const float *__restrict__ gain, float eps, const LiveRows lr) {
  constexpr int RM = MT / 4, RF = FN / 8;
  extern __shared__ __align__(16) float f32_smem[];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int f0 = blockIdx.x * FN, t0 = blockIdx.y * MT;
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (lr.n_live) {
    M = min(M, *reinterpret_cast<const volatile int *>(lr.n_live) * lr.q_len);
    if (t0 >= M) return;
  }
  const int ld = K + 4, vpr = K >> 2;
  float *Ws = f32_smem, *As = f32_smem + FN * ld;
  for (int i = tid; i < FN * vpr; i += 256) {
    const int r = i / vpr, c = (i % vpr) * 4;
    if (f0 + r < N) cp_async16(Ws + r * ld + c, W + (size_t)(f0 + r) * K + c);
    else *reinterpret_cast<float4 *>(Ws + r * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_sync();
  for (int i = tid; i < MT * vpr; i += 256) {
    const int r = i / vpr, c = (i % vpr) * 4;
    if (t0 + r < M) cp_async16(As + r * ld + c, A + (size_t)(t0 + r) * K + c);
    else *reinterpret_cast<float4 *>(As + r * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // the old values of this thread's outputs (residual epilogue), while the copies fly
  constexpr int OUT = MT * FN / 256;                           // outputs per thread, consecutive features
  const int orow = tid * OUT / FN, ocol = tid * OUT % FN;
  const int t = t0 + orow, f = f0 + ocol;
  float old[OUT];
#pragma unroll
  for (int i = 0; i < OUT; ++i) old[i] = (epi == EPI_RESID && t < M && f + i < N) ? C[(size_t)t * N + f + i] : 0.f;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (gain) {
    for (int r = w; r < MT; r += 8) {                          // one warp per row
      float ss = 0.f;
      for (int v = lane; v < vpr; v += 32) {
        const float4 a = *reinterpret_cast<const float4 *>(As + r * ld + v * 4);
        ss = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, ss))));
      }
      const float rstd = rsqrtf(warp_sum(ss) / K + eps);
      for (int v = lane; v < vpr; v += 32) {
        float4 a = *reinterpret_cast<const float4 *>(As + r * ld + v * 4);
        const float4 g = *reinterpret_cast<const float4 *>(gain + v * 4);
        a.x = g.x * a.x * rstd; a.y = g.y * a.y * rstd; a.z = g.z * a.z * rstd; a.w = g.w * a.w * rstd;
        *reinterpret_cast<float4 *>(As + r * ld + v * 4) = a;
      }
    }
    __syncthreads();
  }

  // lane (tr, tf): token rows tr, tr + 4, ..., feature rows tf, tf + 8, ...
  const int tr = lane >> 3, tf = lane & 7;
  float acc[RM][RF];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RF; ++j) acc[i][j] = 0.f;
  for (int v = w; v < vpr; v += 8) {
    float4 a[RM], b[RF];
#pragma unroll
    for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4 *>(As + (tr + 4 * i) * ld + v * 4);
#pragma unroll
    for (int j = 0; j < RF; ++j) b[j] = *reinterpret_cast<const float4 *>(Ws + (tf + 8 * j) * ld + v * 4);
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RF; ++j)
        acc[i][j] = fmaf(a[i].x, b[j].x, fmaf(a[i].y, b[j].y, fmaf(a[i].z, b[j].z, fmaf(a[i].w, b[j].w, acc[i][j]))));
  }
  __syncthreads();                                             // the rows are done with: their space takes the partial tiles
  float *red = f32_smem + w * (MT * FN);
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RF; ++j) red[(tr + 4 * i) * FN + tf + 8 * j] = acc[i][j];
  __syncthreads();
  if (t >= M) return;
#pragma unroll
  for (int i = 0; i < OUT; ++i) {
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += f32_smem[k * (MT * FN) + tid * OUT + i];
    if (f + i < N) C[(size_t)t * N + f + i] = epi == EPI_RESID ? old[i] + v : epi == EPI_GELU_T ? gelu_erf(v) : v;
  }
}

// ------------------------------------------------------------------ host side
// The shapes it takes: rows of which a 32 x 32 tile fits in shared memory (K <= 768: 198 KB), operands
// 16-byte aligned; longer rows keep gemm_simt_kernel.  32 x 32 tiles (twice the flops per shared-memory
// read) where the 16 x 16 ones would be more than one wave at four CTAs per SM.
constexpr int F32_MAX_K = 768;

static int gemm_f32_init() {
  if (cudaFuncSetAttribute(gemm_f32_kernel<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_f32_kernel<32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
    return -4;
  return 0;
}
static bool gemm_f32_eligible(const void *W, int K) { return K % 16 == 0 && K >= 16 && K <= F32_MAX_K && !((uintptr_t)W & 15); }

static bool gemm_f32_launch(cudaStream_t st, bool pdl, const float *A, const float *W, float *C, int M, int N, int K, int epi,
                            const float *gain, float eps, LiveRows lr) {
  const bool small = (long)((N + 15) / 16) * ((M + 15) / 16) <= 4 * 148;
  const int T = small ? 16 : 32;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((N + T - 1) / T, (M + T - 1) / T);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = small ? f32_smem_bytes<16, 16>(K) : f32_smem_bytes<32, 32>(K);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return (small ? cudaLaunchKernelEx(&cfg, gemm_f32_kernel<16, 16>, A, W, C, M, N, K, epi, gain, eps, lr)
                : cudaLaunchKernelEx(&cfg, gemm_f32_kernel<32, 32>, A, W, C, M, N, K, epi, gain, eps, lr)) == cudaSuccess;
}

}  // namespace tsfm
