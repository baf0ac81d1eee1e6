// Small-batch contraction with the weight tile in registers.
//
//   C[t, f] (op)= sum_k A[t, k] * W[f, k]        A: [M, K] tokens (bf16), W: [N, K] weights
//
// For the passes of a few dozen tokens (draft steps, one-token decode steps, short verification
// passes) a contraction is a dependent link in a chain of launches, and what it costs is the
// latency between "my input is ready" and "my output is written".  This kernel keeps that path
// short:
//   * a CTA owns 16 output features x 32 tokens over the WHOLE K range, so nothing is exchanged
//     between CTAs and every epilogue (GELU, residual, folded norm) sees complete sums;
//   * the eight warps split K among them (warp w takes the 64-wide blocks w, w + 8, ...); a lane holds 16
//     consecutive k of a weight row and of a token row, 32 bytes each, straight from global memory in the
//     registers that mma.sync m16n8k16 wants: the contraction does not care which k sits at which of its
//     positions as long as both operands agree, so no shared memory, barrier or ldmatrix stands between the
//     loads and the MMAs, and rows that do not exist are not touched;
//   * the weights do not depend on the preceding kernel: they are in registers BEFORE the dependency wait
//     (programmatic dependent launch);
//   * the partial tiles are summed through shared memory in a fixed order.
// Bound: latency.  A link of a chain of dependent launches, us, with both tiles staged in shared memory -> here:
// M = 1: K = 512 2.5 to 2.7 -> 1.7, K = 2048 4.5 -> 2.3; M = 29: 2.6 to 2.8 -> 1.9 to 2.2, 5.0 -> 3.7; M = 64,
// K = 384: 2.5 to 3.4 -> 1.9 to 2.7.  (A launch that only reads and writes one value per thread: 0.9 to 1.0.)
// The tensor-memory kernels stay the tool wherever K is long, tokens are many or the grid would not fit in one
// wave.
// grid = (ceil(N / 16), ceil(M / 32)), block = 256.  K a multiple of 64, at most WS_MAX_K.
#pragma once
#include "common.cuh"
#include "kernels_simt.cuh"
#include "gemm_sk.cuh"

namespace tsfm {

constexpr int WS_FN = 16, WS_MT = 32, WS_WARPS = 8, WS_MAX_K = 2048;

// (volatile with a memory clobber: stays behind the dependency wait)
__device__ __forceinline__ uint4 ws_ld16(const bf16 *p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// NB: 64-wide blocks of K per warp (at most).  NORM: compile the folded-RMSNorm epilogues (SkNorm; slices of 16
// features).
template <int NB, bool NORM>
__global__ void __launch_bounds__(256, NB == 1 ? 3 : NB == 2 ? 2 : 1)
gemm_ws_kernel(const bf16 *A, const bf16 *__restrict__ W, void *C, int M, int N, int K,
               int epi, const SkNorm nm, const LiveRows lr) {
  __shared__ float red[WS_WARPS * WS_MT * WS_FN], rs[WS_MT];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int f0 = blockIdx.x * WS_FN, t0 = blockIdx.y * WS_MT;
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (lr.n_live) {
    M = min(M, *reinterpret_cast<const volatile int *>(lr.n_live) * lr.q_len);
    if (t0 >= M) return;
  }
  const int KB = K >> 6, g = lane >> 2, q4 = lane & 3;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);

  // ---- weight fragments: independent of the preceding kernel
  uint4 wf[NB][2][2];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int kb = w + b * WS_WARPS, f = f0 + n * 8 + g;
      const bool in = kb < KB && f < N;
      const uint4 *p = reinterpret_cast<const uint4 *>(W + (size_t)f * K + kb * 64 + q4 * 16);
      wf[b][n][0] = in ? __ldg(p) : zero;
      wf[b][n][1] = in ? __ldg(p + 1) : zero;
    }
  // the gains of this thread's two output features (folded norm): constants, fetched before the wait
  float2 gg = make_float2(0.f, 0.f);
  if (NORM && nm.a_out && f0 + (tid & 7) * 2 < N) gg = *reinterpret_cast<const float2 *>(nm.gain + f0 + (tid & 7) * 2);
  pdl_sync();
  // ---- token fragments: rows g and g + 8 of each 16-row tile
  const int n_mt = t0 + 16 < M ? 2 : 1;
  uint4 af[2][NB][2][2];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int kb = w + b * WS_WARPS, t = t0 + m * 16 + r * 8 + g;
        const bool in = kb < KB && t < M;
        const bf16 *p = A + (size_t)t * K + kb * 64 + q4 * 16;
        af[m][b][r][0] = zero;
        af[m][b][r][1] = zero;
        if (in) {
          af[m][b][r][0] = ws_ld16(p);
          af[m][b][r][1] = ws_ld16(p + 8);
        }
      }
  // ---- while the loads fly: this thread's two outputs, their old values, the rows' rstd
  const int orow = tid >> 3, ocol = (tid & 7) * 2;             // output (orow, ocol), (orow, ocol + 1) of the tile
  const int t = t0 + orow, f = f0 + ocol;
  const bool live = t < M && f < N;                            // (N is even: both columns or none)
  float2 old = make_float2(0.f, 0.f);
  if (epi == EPI_RESID && live) old = *reinterpret_cast<const float2 *>((const float *)C + (size_t)t * N + f);
  if (NORM && nm.ssq_in) {
    float acc = 0.f;
    if (t < M) {
      const float4 *src = reinterpret_cast<const float4 *>(nm.ssq_in + (size_t)t * nm.n_part);   // (d % 64 == 0: whole quads)
#pragma unroll 4
      for (int j = tid & 7; j < (nm.n_part >> 2); j += 8) {
        const float4 q = src[j];
        acc += (q.x + q.y) + (q.z + q.w);
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    if ((tid & 7) == 0) rs[orow] = rsqrtf(acc * nm.inv_d + nm.eps);
  }
  // ---- main loop; acc[row tile][feature tile][4]
  float acc[2][2][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b][0] = acc[a][b][1] = acc[a][b][2] = acc[a][b][3] = 0.f;
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    if (m >= n_mt) break;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int s = 0; s < 2; ++s) {                            // 16-byte halves: two k steps each
        const uint4 lo = af[m][b][0][s], hi = af[m][b][1][s];
        const uint32_t a0[4] = {lo.x, hi.x, lo.y, hi.y}, a1[4] = {lo.z, hi.z, lo.w, hi.w};
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          mma_bf16_16816(acc[m][n], a0, wf[b][n][s].x, wf[b][n][s].y);
          mma_bf16_16816(acc[m][n], a1, wf[b][n][s].z, wf[b][n][s].w);
        }
      }
  }
  // ---- partial tiles to shared memory, summed in warp order
  {
    float *mine = red + w * (WS_MT * WS_FN);
    const int q = q4 * 2;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        *reinterpret_cast<float2 *>(mine + (a * 16 + g) * WS_FN + b * 8 + q) = make_float2(acc[a][b][0], acc[a][b][1]);
        *reinterpret_cast<float2 *>(mine + (a * 16 + g + 8) * WS_FN + b * 8 + q) = make_float2(acc[a][b][2], acc[a][b][3]);
      }
  }
  __syncthreads();
  float2 v = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < WS_WARPS; ++i) {
    const float2 p = *reinterpret_cast<const float2 *>(red + i * (WS_MT * WS_FN) + orow * WS_FN + ocol);
    v.x += p.x;
    v.y += p.y;
  }
  // ---- epilogue
  if (NORM && nm.ssq_in) { const float k = rs[orow]; v.x *= k; v.y *= k; }
  const size_t o = (size_t)t * N + f;
  if (epi == EPI_RESID) {
    v.x += old.x;
    v.y += old.y;
    if (live) *reinterpret_cast<float2 *>((float *)C + o) = v;
    if (NORM && nm.a_out) {
      // the next contraction's operand bf16(gain * x) and the row's sum of squares over these 16 features
      if (live) *reinterpret_cast<uint32_t *>(nm.a_out + o) = pack_bf16x2(gg.x * v.x, gg.y * v.y);
      float sq = live ? v.x * v.x + v.y * v.y : 0.f;
      sq += __shfl_xor_sync(0xffffffffu, sq, 1);
      sq += __shfl_xor_sync(0xffffffffu, sq, 2);
      sq += __shfl_xor_sync(0xffffffffu, sq, 4);
      if ((tid & 7) == 0 && t < M && f0 < N) nm.ssq_out[(size_t)t * (N >> 4) + (f0 >> 4)] = sq;
    }
  } else if (live) {
    if (epi == EPI_F32) *reinterpret_cast<float2 *>((float *)C + o) = v;
    else if (epi == EPI_T) *reinterpret_cast<uint32_t *>((bf16 *)C + o) = pack_bf16x2(v.x, v.y);
    else *reinterpret_cast<uint32_t *>((bf16 *)C + o) = pack_bf16x2(gelu_erf_fast(v.x), gelu_erf_fast(v.y));
  }
}

// ------------------------------------------------------------------ host side
static inline int ws_blocks(int K) { return (K / 64 + WS_WARPS - 1) / WS_WARPS; }

// Whether the kernel can serve a shape well: K in the registers of eight warps, N even, the operands 16-byte aligned, and the
// whole grid resident at once -- three CTAs per SM by registers where a warp has one block of K, two with two, else one.
static bool gemm_ws_fits(const void *A, const void *W, int M, int N, int K) {
  if (M < 1 || M > 512 || K < 64 || K % 64 || K > WS_MAX_K || N % 2) return false;
  if (((uintptr_t)A & 15) || ((uintptr_t)W & 15)) return false;
  const int nb = ws_blocks(K), per_sm = nb == 1 ? 3 : nb == 2 ? 2 : 1;
  const long ctas = (long)((N + WS_FN - 1) / WS_FN) * ((M + WS_MT - 1) / WS_MT);
  return ctas <= (long)per_sm * 148;
}
// Whether it is the better one there.  Contractions that do not widen (Wo, W2): where they have less than a million weights or
// fewer than 24 tokens (decode steps of whole models, us a layer, this / gemm_push_kernel: N = K = 1024 M = 20 19.4 / 19.8, 24 21.3 /
// 20.0, 32 21.9 / 20.1, 93 26.4 / 25.1, 128 28.4 / 27.6; N = 512, K = 2048 M = 11 11.5 / 12.4, 24 13.7 / 13.8, 48 17.6 / 16.5, 96
// 18.8 / 18.4; N = K = 2048 M = 24 29.2 / 25.3; N = K = 768 M = 32 21.0 / 22.2, 128 24.5 / 25.6; N = 384, K = 1536 M = 32 14.2 / 14.5;
// in chains of the contraction alone, with weights in L2, N = K = 1024 M = 128 3.7 / 4.1).  Those that widen (QKV,
// W1) scale their rows by factors that every CTA has to sum up: up to 256 CTAs (N = 2048, K = 512: M = 64 3.67 / 3.71, M = 93
// 3.92 / 3.67), and with K > 512 only while the weights come from L2 in time (N = 2304, K = 768: M = 32 3.9 / 4.0; N = 3072, K =
// 1024: M = 8 3.1 / 3.5, M = 16 3.58 / 3.53, M = 24 4.3 / 3.7).
static bool gemm_ws_eligible(const void *A, const void *W, int M, int N, int K) {
  if (!gemm_ws_fits(A, W, M, N, K)) return false;
  if (N <= K) return (long)N * K < 1000000 || M < 24;
  const long ctas = (long)((N + WS_FN - 1) / WS_FN) * ((M + WS_MT - 1) / WS_MT);
  return ws_blocks(K) == 1 ? ctas <= 256 : (long)N * K <= 2500000 || M <= 8;
}

// Shapes that the single-contraction entry point gives to this kernel on request: those that a decoder gives it, and
// up to 256 tokens on up to eight CTAs per SM where K is short (shapes it has always taken; they run in several waves).
static bool gemm_ws_accepts(const void *A, const void *W, int M, int N, int K) {
  if (gemm_ws_fits(A, W, M, N, K)) return true;
  if (M < 1 || M > 256 || K < 64 || K % 64 || K > WS_MAX_K || N % 2) return false;
  if (((uintptr_t)A & 15) || ((uintptr_t)W & 15)) return false;
  const int per_sm = std::min(8, 228 * 1024 / ((WS_FN + WS_MT) * K * 2 + 17536));
  const long ctas = (long)((N + WS_FN - 1) / WS_FN) * ((M + WS_MT - 1) / WS_MT);
  return ctas <= (long)per_sm * 148;
}

static bool gemm_ws_launch(cudaStream_t st, bool pdl, const void *A, const void *W, void *C, int M, int N, int K, int epi,
                           const SkNorm *norm, LiveRows lr) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((N + WS_FN - 1) / WS_FN, (M + WS_MT - 1) / WS_MT);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  const SkNorm nm = norm ? *norm : SkNorm{};
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, (const bf16 *)A, (const bf16 *)W, C, M, N, K, epi, nm, lr) == cudaSuccess;
  };
  switch (ws_blocks(K)) {
    case 1: return norm ? go(gemm_ws_kernel<1, true>) : go(gemm_ws_kernel<1, false>);
    case 2: return norm ? go(gemm_ws_kernel<2, true>) : go(gemm_ws_kernel<2, false>);
    case 3: return norm ? go(gemm_ws_kernel<3, true>) : go(gemm_ws_kernel<3, false>);
    default: return norm ? go(gemm_ws_kernel<4, true>) : go(gemm_ws_kernel<4, false>);
  }
}

}  // namespace tsfm
