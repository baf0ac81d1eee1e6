// fp32 rows x bf16 weights on the tensor cores, exact products: the patch embedding and the mean head of bf16 models.
//
//   C[t, f] = sum_k A'[t, k] * W[f, k]        A' = A, or gain * A / sqrt(mean(A^2) + eps)
//
// A row's values are split into three bf16 parts that add up to them exactly (the leading 8 bits of the mantissa, the next 8, the
// rest: truncation, no rounding), so that three MMAs give the products of the fp32 value.  An MMA cuts its sum off at 24 bits
// instead of rounding it, always towards zero: a chain of them over all of K had 3 to 13 times the error of fp32 FMAs (512 to 2048
// values), so each block of 32 k is summed from zero, the small parts first, and added to the others by an ordinary addition.
//   * a CTA takes 32 rows and 8 NTW wn features; the rows go through in chunks of 256 values: copied to shared memory a chunk
//     ahead, multiplied by the gain, split once, and put back as three tiles that all warps read;
//   * the eight warps are wn groups of 8 NTW features x 8 / wn groups of 32-wide blocks of k (in turn); partial sums of the latter
//     are added through shared memory in a fixed order;
//   * a lane takes 16 consecutive bytes of a weight row and of a row's part as the fragments of two MMAs (which k sits at which
//     position does not matter as long as both operands agree); weights come straight from global memory a block ahead, the first
//     ones before the dependency wait.
// Bound: MMAs (three times the products) and the chain of a CTA for many rows, the round trips of the chunks for few.  fp32 FMAs
// (gemm_f32_kernel's tiles) -> here, us: embedding of 6000 rows of 96, d = 1024 99 -> 34, of 5120, d = 768 60 -> 18, of 16320 rows
// of 32, d = 1280 230 -> 70; head of 6000 rows 68 -> 32, of 5120 52 -> 25, of 1280 26 -> 15, of 576 (d = 1280) 26 -> 14.
// Relative error against 64 bits of both together, layers that add nothing: 1.2e-7 ... 1.8e-7 -> 1.0e-7 ... 1.3e-7.
// grid = (ceil(N / (8 NTW wn)), row tiles), row tiles as in gemm_f32_kernel; block = 256.  K, N multiples of 16.
#pragma once
#include "attn_flash.cuh"
#include "gemm_f32.cuh"

namespace tsfm {

constexpr int GR_ROWS = 32, GR_CHUNK = 256;
// bytes of a row of a part: the eight rows that a warp reads at a time lie 64 bytes apart modulo 128
__host__ __device__ inline int gr_pitch(int KC) { return 2 * KC + (KC & 32 ? 0 : 64); }
inline int gr_chunk(int K) { return K < GR_CHUNK ? (K + 31) & ~31 : GR_CHUNK; }

// The leading bf16 parts of a pair of values, packed, and what is left of the values.
__device__ __forceinline__ uint32_t gr_part(float &a, float &b) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  a -= __uint_as_float(ua & 0xffff0000u);
  b -= __uint_as_float(ub & 0xffff0000u);
  return __byte_perm(ua, ub, 0x7632);
}

template <int NTW>
__global__ void __launch_bounds__(256, 2)
gemm_rows_kernel(const float *A, const bf16 *__restrict__ W, float *C, int M, int N, int K, int wn, const RowsArgs ra) {
  extern __shared__ __align__(16) uint8_t gr_smem[];           // [3 parts][32 rows][pitch], the next chunk [32][KC], gains [K]; at the end partial sums
  __shared__ long long src_off[GR_ROWS], dst_off[GR_ROWS];
  __shared__ int row_series[GR_ROWS];
  __shared__ float row_ss[GR_ROWS];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, q = lane & 3;
  const long long row_tile = (long long)blockIdx.z * F32_GRID_Y + blockIdx.y;
  if (row_tile * GR_ROWS >= M) return;
  const int t0 = (int)row_tile * GR_ROWS, wk = 8 / wn, kg = w / wn;
  const int fw = (blockIdx.x * wn + w % wn) * (8 * NTW);       // first feature of this warp
  const int KC = K < GR_CHUNK ? (K + 31) & ~31 : GR_CHUNK, pitch = gr_pitch(KC);
  const uint32_t parts = (uint32_t)__cvta_generic_to_shared(gr_smem), part_bytes = (uint32_t)(GR_ROWS * pitch);

  // weights of block `blk` (32 k, counted over all of K) of this warp's features
  uint4 wf[NTW];
  auto load_w = [&](int blk) {
    const int k = blk * 32 + 8 * q;
#pragma unroll
    for (int j = 0; j < NTW; ++j) {
      const int f = fw + 8 * j + g;
      wf[j] = f < N && k < K ? __ldg(reinterpret_cast<const uint4 *>(W + (size_t)f * K + k)) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  load_w(kg);
  float *const gains = reinterpret_cast<float *>(gr_smem + 3 * part_bytes + GR_ROWS * KC * 4);
  if (ra.gain)
    for (int k = tid * 4; k < K; k += 1024) *reinterpret_cast<float4 *>(gains + k) = *reinterpret_cast<const float4 *>(ra.gain + k);
  const bool early = !ra.opens_round;
  auto lookup = [&]() {
    if (tid < GR_ROWS) rows_lookup(ra, t0 + tid, M, N, K, &src_off[tid], &dst_off[tid], &row_series[tid]);
  };
  if (early) lookup();
  pdl_sync();
  if (ra.stamp && blockIdx.x == 0 && t0 == 0 && tid == 0) *ra.stamp = globaltimer_ns();
  if (!early) lookup();
  if (!__syncthreads_or(tid < GR_ROWS && src_off[tid] >= 0)) return;     // a tile of dead slots

  // rows 4 w ... 4 w + 3 of a chunk: 16-byte pieces lane and lane + 32, copied and read by the same lane
  float *const chunk = reinterpret_cast<float *>(gr_smem + 3 * part_bytes) + 4 * w * KC;
  auto load_a = [&](int k0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const long long so = src_off[4 * w + r];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int c = (lane + 32 * p) * 4;
        if (c >= KC) continue;
        if (so >= 0 && k0 + c < K) cp_async16(chunk + r * KC + c, A + so + k0 + c);
        else *reinterpret_cast<float4 *>(chunk + r * KC + c) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  load_a(0);
  // a lane's shares of its four rows' sums of squares; between chunks in shared memory where registers are short (with them 48 bytes
  // spilled: embedding of 6000 rows of 96, d = 1024 31.4 -> 30.6 us, of 16000 of 32, d = 1280 69 -> 66.5, head of 5120, d = 768 25.2 -> 24.7)
  __shared__ float4 ss_kept[NTW == 1 ? 1 : 256];
  float acc[2][NTW][4], ss_own[4] = {0.f, 0.f, 0.f, 0.f};
  if (NTW > 1) ss_kept[tid] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < NTW; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;

  for (int k0 = 0; k0 < K; k0 += KC) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (k0) __syncthreads();                                   // the previous chunk's parts are done with
    const float4 so_far = NTW == 1 ? make_float4(ss_own[0], ss_own[1], ss_own[2], ss_own[3]) : ss_kept[tid];
    float ss[4] = {so_far.x, so_far.y, so_far.z, so_far.w};
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int c = (lane + 32 * p) * 4;
      if (c >= KC) continue;
      const float4 gv = ra.gain && k0 + c < K ? *reinterpret_cast<const float4 *>(gains + k0 + c) : make_float4(1.f, 1.f, 1.f, 1.f);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float4 a = *reinterpret_cast<const float4 *>(chunk + r * KC + c);
        if (ra.gain) {
          ss[r] = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, ss[r]))));
          a.x *= gv.x; a.y *= gv.y; a.z *= gv.z; a.w *= gv.w;
        }
        uint8_t *to = gr_smem + (4 * w + r) * pitch + c * 2;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const uint32_t lo = gr_part(a.x, a.y), hi = gr_part(a.z, a.w);
          *reinterpret_cast<uint2 *>(to + s * part_bytes) = make_uint2(lo, hi);
        }
      }
    }
    if (NTW == 1) ss_own[0] = ss[0], ss_own[1] = ss[1], ss_own[2] = ss[2], ss_own[3] = ss[3];
    else ss_kept[tid] = make_float4(ss[0], ss[1], ss[2], ss[3]);
    if (k0 + KC < K) load_a(k0 + KC);                          // flies while this chunk is multiplied
    __syncthreads();
    const int blocks = (min(KC, K - k0) + 31) >> 5, b0 = k0 >> 5;
    for (int b = kg; b < blocks; b += wk) {
      uint4 wc[NTW];
#pragma unroll
      for (int j = 0; j < NTW; ++j) wc[j] = wf[j];
      // the warp's next block: in this chunk, or the first of the next
      if (b + wk < blocks) load_w(b0 + b + wk);
      else load_w(((k0 + KC) >> 5) + kg);
      const uint32_t row = parts + (uint32_t)(g * pitch + b * 64 + q * 16);
      float sum[2][NTW][4];                                    // of this block alone: see above
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int j = 0; j < NTW; ++j) sum[m][j][0] = sum[m][j][1] = sum[m][j][2] = sum[m][j][3] = 0.f;
#pragma unroll
      for (int s = 2; s >= 0; --s) {                           // the small parts first
        uint4 a[2][2];                                         // rows g and g + 8 of each 16
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(a[i >> 1][i & 1].x), "=r"(a[i >> 1][i & 1].y), "=r"(a[i >> 1][i & 1].z), "=r"(a[i >> 1][i & 1].w)
                       : "r"(row + (uint32_t)s * part_bytes + (uint32_t)(8 * i * pitch)) : "memory");
#pragma unroll
        for (int j = 0; j < NTW; ++j)
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const uint32_t a0[4] = {a[m][0].x, a[m][1].x, a[m][0].y, a[m][1].y};
            mma_bf16_16816(sum[m][j], a0, wc[j].x, wc[j].y);
          }
#pragma unroll
        for (int j = 0; j < NTW; ++j)
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const uint32_t a1[4] = {a[m][0].z, a[m][1].z, a[m][0].w, a[m][1].w};
            mma_bf16_16816(sum[m][j], a1, wc[j].z, wc[j].w);
          }
      }
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int j = 0; j < NTW; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[m][j][e] += sum[m][j][e];
    }
  }
  if (ra.gain) {
    const float4 all = NTW == 1 ? make_float4(ss_own[0], ss_own[1], ss_own[2], ss_own[3]) : ss_kept[tid];
    const float ss[4] = {all.x, all.y, all.z, all.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float t = warp_sum(ss[r]);
      if (lane == 0) row_ss[4 * w + r] = t;
    }
  }
  __syncthreads();                                             // the parts are done with: their space takes the partial sums
  float4 *red = reinterpret_cast<float4 *>(gr_smem);           // [kg - 1][m, j][feature group][lane]
  if (kg > 0)
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int j = 0; j < NTW; ++j)
        red[(((kg - 1) * 2 * NTW + m * NTW + j) * wn + w % wn) * 32 + lane] = make_float4(acc[m][j][0], acc[m][j][1], acc[m][j][2], acc[m][j][3]);
  __syncthreads();
  if (kg > 0) return;
  const bool sampled = ra.mode == ROWS_HEAD_LAST && ra.st && (ra.st->flags & VAR_SAMPLE_PROPOSALS);
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < NTW; ++j) {
      for (int k = 0; k < wk - 1; ++k) {
        const float4 p = red[((k * 2 * NTW + m * NTW + j) * wn + w) * 32 + lane];
        acc[m][j][0] += p.x; acc[m][j][1] += p.y; acc[m][j][2] += p.z; acc[m][j][3] += p.w;
      }
      const int f = fw + 8 * j + 2 * q;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = 16 * m + 8 * h + g;
        if (f >= N || src_off[row] < 0) continue;
        const float rstd = ra.gain ? rsqrtf(row_ss[row] / K + ra.eps) : 1.f;
        float v0 = acc[m][j][2 * h] * rstd, v1 = acc[m][j][2 * h + 1] * rstd;
        float *dst = C + dst_off[row] + f;
        if (ra.mode == ROWS_EMBED) {
          *reinterpret_cast<float2 *>(dst) = make_float2(v0, v1);
          continue;
        }
        if (sampled) {     // proposal x = mu_q + sigma_q eps (Sec. 3.3); the mean is kept for the statistic
          float *mu = ra.muq + ((size_t)row_series[row] * ra.Kblk + ra.k_pos) * N + f;
          mu[0] = v0;
          mu[1] = v1;
          v0 += ra.st->sigma_q * head_normal(ra.st, row_series[row], ra.k_pos, f);
          v1 += ra.st->sigma_q * head_normal(ra.st, row_series[row], ra.k_pos, f + 1);
        }
        dst[0] = v0;                                           // (a token may be a single value: no alignment)
        dst[1] = v1;
      }
    }
}

// ------------------------------------------------------------------ host side
struct RowsShape {
  int NTW, wn;
};
// Features per CTA: as many as give the machine a CTA per SM, 8 at least.  Three vectors of eight features per warp where they
// are many, one elsewhere (us, 6000 rows of 96 -> 1024: 192 features a CTA 34, 256 in four vectors 37, 128 in two 41, 64 in one
// 38; heads, 6000 rows of 1024 -> 96: 96 in three vectors 32, 64 in one 53, 32 in one 38; 1280 rows: 16 in one 14.8, in two 22).
static RowsShape gemm_rows_shape(int M, int N) {
  static const RowsShape shapes[] = {{3, 8}, {3, 4}, {1, 8}, {1, 4}, {1, 2}, {1, 1}};         // 192 96 64 32 16 8
  const long rows = (M + GR_ROWS - 1) / GR_ROWS;
  for (int i = 0; i < 5; ++i) {
    const int nt = 8 * shapes[i].NTW * shapes[i].wn, next = 8 * shapes[i + 1].NTW * shapes[i + 1].wn;
    if (next < N && rows * ((N + nt - 1) / nt) >= 148) return shapes[i];
  }
  return shapes[5];
}
static int gemm_rows_smem(int K, bool gain, const RowsShape &s) {
  const int KC = gr_chunk(K), parts = 3 * GR_ROWS * gr_pitch(KC) + GR_ROWS * KC * 4 + (gain ? K * 4 : 0);
  const int red = (8 / s.wn - 1) * 2 * s.NTW * s.wn * 32 * 16;
  return parts > red ? parts : red;
}
static int gemm_rows_init() {
  for (auto *kernel : {gemm_rows_kernel<1>, gemm_rows_kernel<3>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess) return -4;
  return 0;
}
// Rows that 16-byte loads can fetch, gains that fit beside a chunk, features that leave in pairs.
static bool gemm_rows_eligible(const void *W, int N, int K) {
  return K % 16 == 0 && K >= 16 && K <= 32768 && N % 16 == 0 && !((uintptr_t)W & 15);
}

// With K <= 128 and as many 16 x 16 tiles as the machine holds at once gemm_f32_reg_kernel is the shorter link: there is nothing to
// overlap a row's three parts with.  us a link of plain decoding, here / there: heads from d = 64, 256 rows to 32 3.7 / 2.5, 512 to 64 4.0 /
// 2.7, 1000 to 96 (378 tiles) 3.7 / 2.7, 512 to 256 (512) 4.6 / 6.6; from d = 128, 256 to 96 4.1 / 3.9, 1000 to 64 (252) 4.5 / 3.3, 1500 to 64
// (376) 4.2 / 7.2; embedding, 520 rows of 16 to d = 64 3.2 / 1.5, of 64 to 128 (264) 3.5 / 2.7, of 32 to 128, 1000 rows (504) 3.5 / 4.1, of 96
// to 128, 700 rows (352) 3.5 / 5.5.
static bool rows_in_registers(int M, int N, int K) {
  return K <= 128 && (long)((N + 15) / 16) * ((M + 15) / 16) <= (K <= 64 ? 3 : 2) * 148;
}

static bool gemm_rows_launch(cudaStream_t st, bool pdl, const float *A, const bf16 *W, float *C, int M, int N, int K, const RowsArgs &ra) {
  const RowsShape sh = gemm_rows_shape(M, N);
  const int nt = 8 * sh.NTW * sh.wn, row_tiles = (M - 1) / GR_ROWS + 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((N + nt - 1) / nt, std::min(row_tiles, F32_GRID_Y), (row_tiles - 1) / F32_GRID_Y + 1);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = gemm_rows_smem(K, ra.gain != nullptr, sh);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  if (rows_in_registers(M, N, K)) {
    cfg.gridDim = dim3((N + 15) / 16, (M + 15) / 16);
    cfg.dynamicSmemBytes = 0;
    return (K <= 64 ? cudaLaunchKernelEx(&cfg, gemm_f32_reg_kernel<bf16, 2>, A, W, C, M, N, K, ra)
                    : cudaLaunchKernelEx(&cfg, gemm_f32_reg_kernel<bf16, 4>, A, W, C, M, N, K, ra)) == cudaSuccess;
  }
  auto go = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, A, W, C, M, N, K, sh.wn, ra) == cudaSuccess; };
  return sh.NTW == 3 ? go(gemm_rows_kernel<3>) : go(gemm_rows_kernel<1>);
}

}  // namespace tsfm
