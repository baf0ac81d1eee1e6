// Contractions of the fp32 models in fp32 FMAs, patch embedding and mean head among them (with a short K and many rows:
// gemm_simt_kernel, see f32_many).
//
//   C[t, f] (op)= sum_k A'[t, k] * W[f, k]       A' = A, or gain * A / sqrt(mean(A^2) + eps)
//
// For the small fp32 models a contraction is a link of a chain of dependent launches and costs what its
// memory round trips cost; a CTA therefore requests its weight rows before the dependency wait and its
// activation rows in one go behind it, and since it holds the rows it also normalises them (no RMSNorm
// launch in front; large contractions of long rows take one, see run_pass).  For the embedding and the head of passes of many rows it is a matter of reading
// every weight once per tile of rows instead of once per row or eight rows.
//   * tile MT tokens x FN features, K in chunks of KC (all of it in one chunk where that fits); the eight
//     warps take the 4-feature vectors of a chunk in turn (vector w, w + 8, ...), each lane accumulating
//     (MT / 4) x (FN / 8) outputs in registers; the partial tiles are summed through shared memory, so
//     every epilogue sees complete sums.  Vectors of four products are summed before they are added, the eight
//     partial sums as a tree: short chains of additions keep the rounding error of a sum at that of a
//     warp-wide tree;
//   * the norm's factor 1 / sqrt(...) is common to a row: the sums run over gain * A (or over A and gain * W, made before the
//     wait, where K is in one chunk: 0.5 us a link less behind it) and are scaled at the end;
//   * rows are padded by 16 bytes: the four token rows and eight feature rows that a warp reads at a
//     time fall into different banks.
// Bound: latency for small shapes (launch, one L2 round trip, the 8-way sum; 3.5 us a link inside a captured
// forecast where the 64 x 64 tile took 8 to 31 us at M = 37 ... 185, K = 128, 512: forecast of one series
// with the 2-layer d = 128 model 636 -> 260 us, of 37 series 2.55 -> 0.90 ms); for many rows the turns of
// loading, waiting and computing of the three CTAs of an SM (16384 x 3072 x 1024: 25 of 75 TFLOP/s).
// grid = (ceil(N / FN), row tiles), block = 256.  K a multiple of 16.  The row tiles take y first, and z where
// there are more than a grid's y can count (2 million rows in tiles of 32).
#pragma once
#include "common.cuh"
#include "kernels_simt.cuh"

namespace tsfm {

// Where the rows of A come from and where results go.
enum : int {
  ROWS_PLAIN = 0,        // A[t, :], C[t, :] with an epilogue EPI_F32 / EPI_GELU_T / EPI_RESID
  ROWS_EMBED = 1,        // A = token t of the pass in the series' history, C[t, :]
  ROWS_HEAD_LAST = 2,    // A = the last token of slot t, C = the series' history behind the pass (see head_kernel)
  ROWS_HEAD_ALL = 3,     // A = boundary token t of the pass, C = vout[series, boundary, :]
};
struct RowsArgs {
  int mode, epi;
  const float *gain;               // [K] or NULL: no norm
  float eps;
  LiveRows lr;                     // ROWS_PLAIN
  PassGeom g;                      // the other modes
  int opens_round;                 // ROWS_EMBED: the slots are looked up after the wait
  unsigned long long *stamp;       // ROWS_EMBED
  int tok_len;                     // ROWS_HEAD_LAST: values per token; sampled proposals:
  const DevState *st;
  float *muq;
  int k_pos, Kblk;
};

// Offsets of row t in A and C (so -1: no such row) and its series, in the modes other than ROWS_PLAIN: see slot_lookup.
__device__ __forceinline__ void rows_lookup(const RowsArgs &ra, int t, int M, int N, int K, long long *so, long long *dof, int *series) {
  const PassGeom &g = ra.g;
  *so = -1;
  *dof = 0;
  if (t >= M) return;
  const int nb = ra.mode == ROWS_HEAD_LAST ? 1 : ra.mode == ROWS_HEAD_ALL ? g.q_len / g.head_step : g.q_len;   // rows per slot
  const int slot = t / nb, i = t % nb;
  const SlotPos sp = slot_lookup(g, slot);
  if (sp.dead) return;
  *series = sp.b;
  if (ra.mode == ROWS_EMBED) {
    *so = ((long long)sp.b * g.cap + sp.p0 + i) * K;
    *dof = (long long)t * N;
    return;
  }
  const int j = ra.mode == ROWS_HEAD_LAST ? g.q_len - 1 : (i + 1) * g.head_step - 1;
  *so = ((long long)slot * g.q_len + j) * K;
  *dof = ra.mode == ROWS_HEAD_LAST ? ((long long)sp.b * g.cap + sp.p0 + g.q_len) * ra.tok_len : ((long long)sp.b * nb + i) * N;
}

constexpr int F32_GRID_Y = 65535;                              // the largest y of a grid

template <int MT, int FN> constexpr int f32_smem_bytes(int KC) {
  const int rows = MT * (KC + 4) * 4 + FN * (KC + 4) * 4, red = 8 * MT * FN * 4;   // the partial sums reuse the rows
  return rows > red ? rows : red;
}

__device__ __forceinline__ float4 f32_vec4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 f32_vec4(const bf16 *p) {
  const uint2 u = *reinterpret_cast<const uint2 *>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}

template <int MT, int FN>
__global__ void __launch_bounds__(256)
gemm_f32_kernel(const float *A, const float *__restrict__ W, float *C, int M, int N, int K, int KC, const RowsArgs ra) {
  constexpr int RM = MT / 4, RF = FN / 8;
  extern __shared__ __align__(16) float f32_smem[];
  __shared__ long long src_off[MT], dst_off[MT];               // row offsets in A and C; src -1: no such row
  __shared__ int row_series[MT];
  __shared__ float row_ss[MT];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long long row_tile = (long long)blockIdx.z * F32_GRID_Y + blockIdx.y;
  if (row_tile * MT >= M) return;                              // (the last z's share of y is not full)
  const int f0 = blockIdx.x * FN, t0 = (int)row_tile * MT;
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (ra.mode == ROWS_PLAIN) {
    if (ra.lr.n_live) M = min(M, *reinterpret_cast<const volatile int *>(ra.lr.n_live) * ra.lr.q_len);
    if (t0 >= M) return;
  }
  auto lookup = [&]() {
    if (tid < MT) rows_lookup(ra, t0 + tid, M, N, K, &src_off[tid], &dst_off[tid], &row_series[tid]);
  };
  const int lda = KC + 4;
  float *As = f32_smem;
  float *Ws = f32_smem + MT * lda;
  auto load_w = [&](int k0, int kc) {
    const int cpr = kc / 4;
    for (int i = tid; i < FN * cpr; i += 256) {
      const int r = i / cpr, c = (i % cpr) * 4;
      if (f0 + r < N) cp_async16(Ws + r * lda + c, W + (size_t)(f0 + r) * K + k0 + c);
      else *reinterpret_cast<float4 *>(Ws + r * lda + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load_w(0, min(KC, K));
  // a norm's gain, where all of K is here at once (and the grid, of small tiles, starts early): multiplied into the weights before the dependency wait, so that behind it the
  // rows are used as they arrive (their sums of squares are not needed before the end)
  const bool gain_in_w = MT == 16 && ra.gain && KC >= K;
  if (gain_in_w) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int vpr = K >> 2;
    for (int i = tid; i < FN * vpr; i += 256) {
      const int r = i / vpr, c = (i - r * vpr) * 4;
      float4 v = *reinterpret_cast<const float4 *>(Ws + r * lda + c);
      const float4 gg = *reinterpret_cast<const float4 *>(ra.gain + c);
      v.x *= gg.x; v.y *= gg.y; v.z *= gg.z; v.w *= gg.w;
      *reinterpret_cast<float4 *>(Ws + r * lda + c) = v;
    }
  }
  const bool early = ra.mode != ROWS_PLAIN && !ra.opens_round;
  if (ra.mode == ROWS_PLAIN) {
    if (tid < MT) {
      src_off[tid] = t0 + tid < M ? (long long)(t0 + tid) * K : -1;
      dst_off[tid] = (long long)(t0 + tid) * N;
    }
  } else if (early) {
    lookup();
  }
  if (tid < MT) row_ss[tid] = 0.f;
  pdl_sync();
  if (ra.stamp && blockIdx.x == 0 && t0 == 0 && tid == 0) *ra.stamp = globaltimer_ns();
  if (ra.mode != ROWS_PLAIN && !early) lookup();
  if (!__syncthreads_or(tid < MT && src_off[tid] >= 0)) {      // a tile of dead slots
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }

  // this thread's outputs: consecutive features of one row; their old values (residual epilogue) fly with the copies
  constexpr int OUT = MT * FN / 256;
  const int orow = tid * OUT / FN, f = f0 + tid * OUT % FN;
  const bool live = src_off[orow] >= 0;
  float *dst = C + dst_off[orow];
  float old[OUT];
#pragma unroll
  for (int i = 0; i < OUT; ++i) old[i] = (ra.epi == EPI_RESID && live && f + i < N) ? dst[f + i] : 0.f;

  // lane (tr, tf): token rows tr, tr + 4, ..., feature rows tf, tf + 8, ...
  const int tr = lane >> 3, tf = lane & 7;
  float acc[RM][RF];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RF; ++j) acc[i][j] = 0.f;
  for (int k0 = 0; k0 < K; k0 += KC) {
    const int kc = min(KC, K - k0), vpr = kc >> 2;
    if (k0) {
      __syncthreads();                                         // the previous chunk is done with
      load_w(k0, kc);
    }
    for (int i = tid; i < MT * vpr; i += 256) {
      const int r = i / vpr, c = (i % vpr) * 4;
      if (src_off[r] >= 0) cp_async16(As + r * lda + c, A + src_off[r] + k0 + c);
      else *reinterpret_cast<float4 *>(As + r * lda + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (ra.gain) {
      for (int r = w; r < MT; r += 8) {                        // one warp per row
        float ss = 0.f;
        for (int v = lane; v < vpr; v += 32) {
          float4 a = *reinterpret_cast<const float4 *>(As + r * lda + v * 4);
          ss = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, ss))));
          if (gain_in_w) continue;
          const float4 gg = *reinterpret_cast<const float4 *>(ra.gain + k0 + v * 4);
          a.x *= gg.x; a.y *= gg.y; a.z *= gg.z; a.w *= gg.w;
          *reinterpret_cast<float4 *>(As + r * lda + v * 4) = a;
        }
        ss = warp_sum(ss);
        if (lane == 0) row_ss[r] += ss;
      }
      if (!gain_in_w) __syncthreads();
    }
    for (int v = w; v < vpr; v += 8) {
      float4 a[RM], b[RF];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4 *>(As + (tr + 4 * i) * lda + v * 4);
#pragma unroll
      for (int j = 0; j < RF; ++j) b[j] = f32_vec4(Ws + (tf + 8 * j) * lda + v * 4);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RF; ++j)
          acc[i][j] += fmaf(a[i].x, b[j].x, fmaf(a[i].y, b[j].y, fmaf(a[i].z, b[j].z, a[i].w * b[j].w)));
    }
  }
  __syncthreads();                                             // the rows are done with: their space takes the partial tiles
  float *red = f32_smem + w * (MT * FN);
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RF; ++j) red[(tr + 4 * i) * FN + tf + 8 * j] = acc[i][j];
  __syncthreads();
  if (!live) return;
  const float rstd = ra.gain ? rsqrtf(row_ss[orow] / K + ra.eps) : 1.f;
  const bool sampled = ra.mode == ROWS_HEAD_LAST && ra.st && (ra.st->flags & VAR_SAMPLE_PROPOSALS);
#pragma unroll
  for (int i = 0; i < OUT; ++i) {
    if (f + i >= N) break;
    float p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = f32_smem[k * (MT * FN) + tid * OUT + i];
    float v = (((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]))) * rstd;
    if (ra.epi == EPI_RESID) v += old[i];
    else if (ra.epi == EPI_GELU_T) v = gelu_erf(v);
    if (sampled) {     // proposal x = mu_q + sigma_q eps (Sec. 3.3); the mean is kept for the statistic
      ra.muq[((size_t)row_series[orow] * ra.Kblk + ra.k_pos) * N + f + i] = v;
      v += ra.st->sigma_q * head_normal(ra.st, row_series[orow], ra.k_pos, f + i);
    }
    dst[f + i] = v;
  }
}

// The same for small grids and short K, 16 x 16 outputs a CTA: a warp's share of K (every eighth vector of four) is nobody else's, so
// both operands go straight into registers, the weights (times a norm's gain) before the dependency wait and all of the rows
// behind it in one round trip; no copy through shared memory and no barrier stands before the sum of the partial tiles.
// Bound: one round trip to L2 and the sum of eight partial tiles.  Links of the fp32 models' forecasts, us, gemm_f32_kernel -> here:
// K = 64 2.3 .. 2.9 -> 1.5 .. 2.1, K = 128 2.0 .. 3.6 -> 1.5 .. 2.8; a speculative forecast of one series 231 -> 207 us,
// of 37 series of different lengths 707 -> 654.  Where it is taken: f32_in_registers; embedding and head of bf16 models (T): rows_in_registers.
// NV: vectors per warp, K <= 32 NV.  grid as above (z = 1), block = 256.
template <typename T, int NV>
__global__ void __launch_bounds__(256, NV <= 2 ? 3 : 2)
gemm_f32_reg_kernel(const float *A, const T *__restrict__ W, float *C, int M, int N, int K, const RowsArgs ra) {
  __shared__ float red[8][256], row_ss[8][16];
  __shared__ long long src_off[16], dst_off[16];               // (modes other than ROWS_PLAIN)
  __shared__ int row_series[16];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, tr = lane >> 3, tf = lane & 7;
  const int f0 = blockIdx.x * 16, t0 = blockIdx.y * 16, orow = tid >> 4, f = f0 + (tid & 15);
  const bool plain = ra.mode == ROWS_PLAIN;
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (plain) {
    if (ra.lr.n_live) M = min(M, *reinterpret_cast<const volatile int *>(ra.lr.n_live) * ra.lr.q_len);
    if (t0 >= M) return;
  }
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 b[NV][2];                                             // features tf, tf + 8
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int k = (w + 8 * n) * 4;
#pragma unroll
    for (int j = 0; j < 2; ++j) b[n][j] = k < K && f0 + tf + 8 * j < N ? f32_vec4(W + (size_t)(f0 + tf + 8 * j) * K + k) : zero;
  }
  if (ra.gain) {
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int k = (w + 8 * n) * 4;
      const float4 gg = k < K ? *reinterpret_cast<const float4 *>(ra.gain + k) : zero;
#pragma unroll
      for (int j = 0; j < 2; ++j) b[n][j].x *= gg.x, b[n][j].y *= gg.y, b[n][j].z *= gg.z, b[n][j].w *= gg.w;
    }
  }
  const bool early = !plain && !ra.opens_round;
  auto lookup = [&]() {
    if (tid < 16) rows_lookup(ra, t0 + tid, M, N, K, &src_off[tid], &dst_off[tid], &row_series[tid]);
  };
  if (early) lookup();
  pdl_sync();
  if (ra.stamp && blockIdx.x == 0 && t0 == 0 && tid == 0) *ra.stamp = globaltimer_ns();
  if (!plain) {
    if (!early) lookup();
    if (!__syncthreads_or(tid < 16 && src_off[tid] >= 0)) return;        // a tile of dead slots
  }
  auto src = [&](int r) { return !plain ? src_off[r] : t0 + r < M ? (long long)(t0 + r) * K : -1ll; };
  float4 a[4][NV];                                             // rows tr, tr + 4, ...
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long so = src(tr + 4 * i);
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int k = (w + 8 * n) * 4;
      a[i][n] = so >= 0 && k < K ? __ldcg(reinterpret_cast<const float4 *>(A + so + k)) : zero;
    }
  }
  const bool live = src(orow) >= 0 && f < N;
  float *dst = C + (plain ? (long long)(t0 + orow) * N : dst_off[orow]) + f;
  const float old = ra.epi == EPI_RESID && live ? __ldcg(dst) : 0.f;
  float acc[4][2], ss[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[i][0] = acc[i][1] = ss[i] = 0.f;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const float4 v = a[i][n];
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] += fmaf(v.x, b[n][j].x, fmaf(v.y, b[n][j].y, fmaf(v.z, b[n][j].z, v.w * b[n][j].w)));
      if (ra.gain) ss[i] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss[i]))));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) red[w][(tr + 4 * i) * 16 + tf + 8 * j] = acc[i][j];
    if (ra.gain && tf == 0) row_ss[w][tr + 4 * i] = ss[i];
  }
  __syncthreads();
  if (!live) return;
  float p[8], q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) p[k] = red[k][tid];
  float v = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
  if (ra.gain) {
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = row_ss[k][orow];
    v *= rsqrtf((((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]))) / K + ra.eps);
  }
  if (ra.epi == EPI_RESID) v += old;
  else if (ra.epi == EPI_GELU_T) v = gelu_erf(v);
  if (ra.mode == ROWS_HEAD_LAST && ra.st && (ra.st->flags & VAR_SAMPLE_PROPOSALS)) {   // (see gemm_f32_kernel)
    ra.muq[((size_t)row_series[orow] * ra.Kblk + ra.k_pos) * N + f] = v;
    v += ra.st->sigma_q * head_normal(ra.st, row_series[orow], ra.k_pos, f);
  }
  *dst = v;
}

// ------------------------------------------------------------------ host side
static int gemm_f32_init() {
  if (cudaFuncSetAttribute(gemm_f32_kernel<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_f32_kernel<32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess)
    return -4;
  return 0;
}
// Rows that 16-byte copies can fetch.
static bool gemm_f32_eligible(const void *W, int K) { return K % 16 == 0 && K >= 16 && !((uintptr_t)W & 15); }

// 16 x 16 tiles where the grid has at most four of them per SM (with rows of 512 fp32 values three fit at a time: the
// largest such grids run somewhat over one wave); beyond that 32 x 32 ones (twice the flops per
// shared-memory read).
static bool gemm_f32_small(int M, int N) { return (long)((N + 15) / 16) * ((M + 15) / 16) <= 4 * 148; }
// Which links take the registers: those of few rows in models of width up to 128.  A CTA of NV = 4 holds half of an SM's
// registers, and past 64 rows the links around it, waiting beside it with their weights, no longer find room (plain decoding,
// 2 layers, d = 128, us a forecast of eight patches, gemm_f32_kernel -> here: 8 series 315 -> 280, 37 356 -> 326, 64 396 -> 384;
// 80 series 406 -> 421, 128 468 -> 499, 256 590 -> 670); NV = 2 a quarter (4 layers, d = 64: 30 series 539 -> 485, 100 604 -> 545,
// 160 666 -> 642; 200 702 -> 721, 700 1241 -> 1281).  The embedding of a wider model alone gives nothing (d = 256: 8 series 475 both,
// 64 735 -> 757), and neither did K = 256 in twice the warps (3.7 us a link for 3.0: more of the time before the wait is weights).
static bool f32_in_registers(int mode, int M, int N, int K) {
  return K <= 128 && (mode != ROWS_EMBED || N <= 128) && M <= (K <= 64 ? 160 : 64);
}
// A small grid keeps rows of up to 768 values whole (one memory round trip), and so does one of up to two 32 x 32 tiles
// per SM with rows of up to 512.  Otherwise rows longer than 256 go through in chunks of 256: three CTAs of 66 KB share an SM,
// one loading while another computes, where rows of 512 in one piece leave room for one
// (2048 x 512 x 512, 1024 CTAs: 68 -> 50 us; 256 x 1536 x 512, 384 CTAs: 29 -> 22; 512 x 512 x 512, 256 CTAs: 19.4 whole,
// 20.7 in chunks).
static bool gemm_f32_launch(cudaStream_t st, bool pdl, const float *A, const float *W, float *C, int M, int N, int K, const RowsArgs &ra) {
  const bool small = gemm_f32_small(M, N);
  const int tile = small ? 16 : 32;
  const bool two_waves = (long)((N + 31) / 32) * ((M + 31) / 32) <= 2 * 148;
  const int KC = K <= (small ? 768 : two_waves ? 512 : 256) ? K : 256;
  cudaLaunchConfig_t cfg{};
  const int row_tiles = (M - 1) / tile + 1;
  cfg.gridDim = dim3((N + tile - 1) / tile, std::min(row_tiles, F32_GRID_Y), (row_tiles - 1) / F32_GRID_Y + 1);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = small ? f32_smem_bytes<16, 16>(KC) : f32_smem_bytes<32, 32>(KC);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  if (small && f32_in_registers(ra.mode, M, N, K)) {
    cfg.dynamicSmemBytes = 0;
    return (K <= 64 ? cudaLaunchKernelEx(&cfg, gemm_f32_reg_kernel<float, 2>, A, W, C, M, N, K, ra)
                    : cudaLaunchKernelEx(&cfg, gemm_f32_reg_kernel<float, 4>, A, W, C, M, N, K, ra)) == cudaSuccess;
  }
  return (small ? cudaLaunchKernelEx(&cfg, gemm_f32_kernel<16, 16>, A, W, C, M, N, K, KC, ra)
                : cudaLaunchKernelEx(&cfg, gemm_f32_kernel<32, 32>, A, W, C, M, N, K, KC, ra)) == cudaSuccess;
}

}  // namespace tsfm
