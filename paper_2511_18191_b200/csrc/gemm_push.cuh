// bf16 x bf16 -> fp32 contraction of up to 512 tokens on the tensor cores (tcgen05), K split over a cluster where it is long.
//
//   C[t, f] (op)= sum_k A[t, k] * W[f, k]        A: [M, K] tokens, W: [N, K] weights
//
// Such a contraction is a link of a chain of dependent launches (one-token decoding and verification of a few dozen
// series), and what it costs is the latency between "my input is ready" and "my output is written", plus the fill of
// the weights that have not arrived by then.  Stamps of every step (%globaltimer, in an instrumented copy) gave what is
// built here:
//   * weight tile 128 features (the MMA's M) x BN tokens (its N); K is split over the S CTAs of a cluster only where
//     its block steps (0.11 us each) outweigh the exchange of the partial tiles (1.2 us);
//   * partial tiles are PUSHED: a thread holds 16 tokens of one feature after tcgen05.ld and sends four of them at a time
//     (st.async, 16 bytes) into the shared memory of the rank that finishes these tokens, whose barrier counts the
//     bytes.  One hop instead of a cluster barrier, a pull through distributed shared memory and a second barrier
//     (0.5 + 1.2 + 0.8 us); sums are taken in rank order, so results do not depend on arrival.  Without a split the
//     epilogue works on the registers;
//   * the epilogue runs on eight warps (got -> done 1.8 us with four, 0.6 with eight and the instantiation per epilogue);
//   * the producer initialises its barriers lane by lane and requests the first ring-full of weights at once, before
//     the dependency wait and before tensor memory is allocated; the rings of weights and tokens are separate, so that
//     a CTA can hold more weights than tokens;
//   * the MMA warp runs its loop as a whole and lets one lane issue: addresses and descriptors are then uniform
//     values (0.21 -> 0.17 us a block step); stages are two K blocks (-> 0.11).
// Bound: latency, and from K = 1280 on the weights (d = 1280, M = 64 from HBM: 39 MB a layer, 6.1 us).  Inside a forecast
// (d = 1280, M = 64, weights from HBM), us a launch, gemm_sk_kernel's former form for these sizes (32-token tiles, K split until the
// grid fills the SMs, pulled partial tiles) -> here, QKV / Wo / W1 / W2: 6.9 / 5.0 / 8.0 / 7.8 -> 5.5 / 5.0 / 5.3 / 7.4: Wo gains
// nothing there.  Chains of these contractions alone (graph replay): d = 1280, M = 64 6.3 / 5.3 / 7.9 / 7.7 -> 5.2 / 4.0 / 6.1 / 6.6;
// d = 1024, M = 93 6.2 / - / 7.1 / 7.0 -> 4.5 / - / 5.4 / 5.9; d = 512, M = 160 5.4 / - / 6.1 / 5.9 -> 3.6 / - / 4.0 / 4.8; d = 1280,
// M = 512 20 / 11 / 31 / 28 -> 9.8 / 8.6 / 12 / 15.  (64-feature tiles: 0.2 % on average, not kept.  A bulk prefetch of the next
// link's weights into L2: nothing.)
// Warps 0-7 epilogue, 8 TMA producer, 9 tensor memory and MMA issue.  Waits are bounded as in gemm_tc.cuh.
#pragma once
#include "gemm_sk.cuh"
#include "gemm_pair.cuh"

namespace tsfm {

constexpr int PUSH_EPI_WARPS = 8, PUSH_THREADS = 32 * (PUSH_EPI_WARPS + 2);
constexpr int PUSH_KS = 2, PUSH_MAX_STAGES = 6, PUSH_MAX_BN = 128;   // K blocks per stage; ring depth; tokens per tile

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// EPI: EPI_F32 / EPI_GELU_T (both scale their rows where nm.ssq_in is given) / EPI_RESID (emits the next norm's operand and sums
// of squares over 16 features where nm.a_out is given).  RB: tokens that a rank finishes (a multiple of 4); SW, SA: stages of
// the weights' and the tokens' ring (SA <= SW).
// grid = (ceil(N / 128), ceil(M / BN), S), cluster = (1, 1, S).
template <int EPI>
__global__ void __launch_bounds__(PUSH_THREADS)
gemm_push_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapA, void *C, int M, int N, int K,
                 int BN, int RB, int SW, int SA, int tmem_cols, const SkNorm nm, int *__restrict__ status, const LiveRows lr) {
  constexpr int W_BLOCK = TC_BM * TC_BK * 2, W_STAGE = PUSH_KS * W_BLOCK;
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (lr.n_live) {
    M = min(M, *reinterpret_cast<const volatile int *>(lr.n_live) * lr.q_len);
    if ((int)blockIdx.y * BN >= M) return;
  }
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int S = gridDim.z, rank = blockIdx.z;
  const int a_block = BN * TC_BK * 2, a_stage = PUSH_KS * a_block;
  const uint32_t tiles_a = tiles + (uint32_t)(SW * W_STAGE);
  const uint32_t recv0 = tiles_a + (uint32_t)(SA * a_stage);                // [source][quad of tokens][feature] x 4 tokens
  const uint32_t bars = recv0 + (uint32_t)(S > 1 ? S * RB * TC_BM * 4 : 0);
  const uint32_t wfirst = bars, accum = bars + 8, recv_bar = bars + 16, slot = bars + 24, wfull0 = bars + 32, afull0 = bars + 80, done0 = bars + 128;
  uint32_t *slot_ptr = reinterpret_cast<uint32_t *>(smem_raw + (slot - smem_u32(smem_raw)));
  float *rs = reinterpret_cast<float *>(smem_raw + (bars + 192 - smem_u32(smem_raw)));
  const float4 *recv = reinterpret_cast<const float4 *>(smem_raw + (recv0 - smem_u32(smem_raw)));

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int f0 = blockIdx.x * TC_BM, t0 = blockIdx.y * BN;
  const int KB_all = (K + TC_BK - 1) / TC_BK;
  const int kb_lo = KB_all * rank / S, KB = KB_all * (rank + 1) / S - kb_lo;
  const int RBQ = RB >> 2;                                                  // token quads per rank
  const int n_quads = (min(M - t0, BN) + 3) >> 2;                           // quads in use
  const int own = min(max(n_quads - rank * RBQ, 0), RBQ);                   // of this rank

  uint32_t tmem = 0;
  const int n_st = (KB + PUSH_KS - 1) / PUSH_KS;                            // stages of this rank's share of K
  if (warp == PUSH_EPI_WARPS) {
    // ---------------- TMA producer: barriers, then the first ring-full of weights (they do not depend on the kernel
    // before), then, behind the dependency wait, the token tiles
    const bool leader = elect_one();
    if (lane < 3) mbar_init(bars + 8 * lane, 1);                            // wfirst, accum, recv_bar
    if (lane < 3 * PUSH_MAX_STAGES) mbar_init(wfull0 + 8 * lane, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    const int pre_w = min(n_st, SW), pre_a = min(n_st, SA);
    if (leader) {
      const int nb = min(KB, pre_w * PUSH_KS);
      mbar_expect_tx(wfirst, (uint32_t)(nb * W_BLOCK));
      for (int kb = 0; kb < nb; ++kb) tma_load_2d(tiles + kb * W_BLOCK, &mapW, (kb_lo + kb) * TC_BK, f0, wfirst);
      mbar_expect_tx(recv_bar, (uint32_t)(own * TC_BM * 16 * (S - 1)));
      for (int st = 0; st < pre_a; ++st) mbar_expect_tx(afull0 + 8 * st, (uint32_t)(min(PUSH_KS, KB - st * PUSH_KS) * a_block));
    }
    __syncwarp();
    asm volatile("bar.arrive 2, %0;" ::"n"(PUSH_THREADS) : "memory");
    if (S > 1) cluster_arrive();
    pdl_sync();
    if (leader) {
      const int nb = min(KB, pre_a * PUSH_KS);
      for (int kb = 0; kb < nb; ++kb) tma_load_2d(tiles_a + kb * a_block, &mapA, (kb_lo + kb) * TC_BK, t0, afull0 + 8 * (kb / PUSH_KS));
    }
    int s = 0, sw = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int st = 0; st + SA < n_st && ok; ++st) {
      ok = mbar_wait(done0 + 8 * s, ph);
      if (!ok) atomicExch(status, DEV_TIMEOUT_TMA);
      if (leader && ok) {
        const int kb = (st + SA) * PUSH_KS, nb = min(PUSH_KS, KB - kb);
        mbar_expect_tx(afull0 + 8 * s, (uint32_t)(nb * a_block));
        for (int i = 0; i < nb; ++i) tma_load_2d(tiles_a + s * a_stage + i * a_block, &mapA, (kb_lo + kb + i) * TC_BK, t0, afull0 + 8 * s);
        if (st + SW < n_st) {
          const int kw = (st + SW) * PUSH_KS, nw = min(PUSH_KS, KB - kw);
          mbar_expect_tx(wfull0 + 8 * sw, (uint32_t)(nw * W_BLOCK));
          for (int i = 0; i < nw; ++i) tma_load_2d(tiles + sw * W_STAGE + i * W_BLOCK, &mapW, (kb_lo + kw + i) * TC_BK, f0, wfull0 + 8 * sw);
        }
      }
      if (++s == SA) { s = 0; ph ^= 1u; }
      if (++sw == SW) sw = 0;
    }
    __syncwarp();
    if (S > 1) { cluster_wait(); cluster_arrive(); }
  } else if (warp == PUSH_EPI_WARPS + 1) {
    // ---------------- tensor memory and MMA issue.  The whole warp runs the loop, so that its addresses and
    // descriptors are uniform values; one lane issues.
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"((uint32_t)tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
    asm volatile("bar.sync 2, %0;" ::"n"(PUSH_THREADS) : "memory");
    tc_fence_after();
    if (S > 1) cluster_arrive();
    tmem = *slot_ptr;
    const bool leader = elect_one();
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
    pdl_sync();
    const uint64_t dw0 = umma_smem_desc(tiles), da0 = umma_smem_desc(tiles_a);
    uint64_t dw = dw0, da = da0;
    int s = 0, sw = 0;
    uint32_t ph = 0, phw = 1;
    bool ok = mbar_wait(wfirst, 0);
    if (!ok) atomicExch(status, DEV_TIMEOUT_MMA);
    for (int st = 0; st < n_st && ok; ++st) {
      if (st >= SW) ok = mbar_wait(wfull0 + 8 * sw, phw);
      if (ok) ok = mbar_wait(afull0 + 8 * s, ph);
      if (!ok) atomicExch(status, DEV_TIMEOUT_MMA);
      if (leader && ok) {
        const uint64_t da1 = da + (uint32_t)(a_block >> 4);
#pragma unroll
        for (int k = 0; k < TC_BK / 16; ++k) umma_bf16(tmem, dw + 2 * k, da + 2 * k, idesc, (st | k) ? 1u : 0u);
        if (2 * st + 1 < KB) {
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k) umma_bf16(tmem, dw + (W_BLOCK >> 4) + 2 * k, da1 + 2 * k, idesc, 1u);
        }
        if (st + SA < n_st) umma_commit(done0 + 8 * s);
      }
      dw += W_STAGE >> 4;
      da += (uint32_t)(a_stage >> 4);
      if (++s == SA) { s = 0; ph ^= 1u; da = da0; }
      if (++sw == SW) { sw = 0; phw ^= 1u; dw = dw0; }
    }
    if (leader && ok) umma_commit(accum);
    __syncwarp();
    if (S > 1) { cluster_wait(); cluster_arrive(); }
  } else {
    const int grp = warp >> 2, w4 = warp & 3;                               // two groups of four warps share the tokens
    const int fl = w4 * 32 + lane, f = f0 + fl, tr = t0 + rank * RB;   // first token of this rank
    const bool mine = f < N;
    asm volatile("bar.sync 2, %0;" ::"n"(PUSH_THREADS) : "memory");
    tc_fence_after();
    if (S > 1) cluster_arrive();
    tmem = *slot_ptr;
    float gain = 0.f;
    if (EPI == EPI_RESID && nm.a_out && f < N) gain = nm.gain[f];
    pdl_sync();
    // old residual values of this thread's first two quads of tokens
    float old[8];
    auto fetch_old = [&](int q0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int q = q0 + 2 * (i >> 2), t = tr + 4 * q + (i & 3);
        old[i] = q < own && mine && t < M ? __ldcg((const float *)C + (size_t)t * N + f) : 0.f;
      }
    };
    if (EPI == EPI_RESID) fetch_old(S > 1 ? grp : 4 * grp);
    if (EPI != EPI_RESID && nm.ssq_in) {
      // eight threads per row, four 16-byte loads in flight each (512 features; longer rows in several rounds)
      const int n4 = nm.n_part >> 2, part = threadIdx.x & 7;
      for (int i = threadIdx.x >> 3; i < 4 * own; i += 32) {
        float acc = 0.f;
        if (tr + i < M) {
          const float4 *src = reinterpret_cast<const float4 *>(nm.ssq_in + (size_t)(tr + i) * nm.n_part);
          for (int j = part; j < n4; j += 32) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = j + 8 * u < n4 ? __ldcg(src + j + 8 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += (v[u].x + v[u].y) + (v[u].z + v[u].w);
          }
        }
        const unsigned m8 = 0xffu << (lane & 24);
        acc += __shfl_xor_sync(m8, acc, 1);
        acc += __shfl_xor_sync(m8, acc, 2);
        acc += __shfl_xor_sync(m8, acc, 4);
        if (part == 0) rs[i] = rsqrtf(acc * nm.inv_d + nm.eps);
      }
      __syncwarp();
      if (S == 1) asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    // Epilogue of the tokens of quads q0 and q0 + 2 (this thread's feature).
    auto finish = [&](int q0, float (&v)[8]) {
      const bool two = q0 + 2 < own;
      if (EPI != EPI_RESID && nm.ssq_in) {
        const float4 k = *reinterpret_cast<const float4 *>(rs + 4 * q0);
        v[0] *= k.x; v[1] *= k.y; v[2] *= k.z; v[3] *= k.w;
        if (two) {
          const float4 k2 = *reinterpret_cast<const float4 *>(rs + 4 * q0 + 8);
          v[4] *= k2.x; v[5] *= k2.y; v[6] *= k2.z; v[7] *= k2.w;
        }
      }
      const int t = tr + 4 * q0;
      const int lim = mine ? min(M - t, two ? 12 : 4) : 0;                  // rows t + 0..3, t + 8..11
      const size_t o = (size_t)t * N + f;
      if (EPI == EPI_F32) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if ((i & 3) + 2 * (i & 4) < lim) ((float *)C)[o + (size_t)((i & 3) + 2 * (i & 4)) * N] = v[i];
      } else if (EPI == EPI_GELU_T) {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          const uint32_t u = gelu_erf_fast2(v[i], v[i + 1]);
          const int d = (i & 3) + 2 * (i & 4);
          if (d < lim) ((uint16_t *)C)[o + (size_t)d * N] = (uint16_t)u;
          if (d + 1 < lim) ((uint16_t *)C)[o + (size_t)(d + 1) * N] = (uint16_t)(u >> 16);
        }
      } else {
        float sq[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int d = (i & 3) + 2 * (i & 4);
          v[i] += old[i];
          if (d < lim) ((float *)C)[o + (size_t)d * N] = v[i];
          if (d < lim && nm.a_out) nm.a_out[o + (size_t)d * N] = __float2bfloat16_rn(gain * v[i]);
          sq[i] = d < lim ? v[i] * v[i] : 0.f;
        }
        if (nm.a_out) {
          // sums over the 16 lanes of a slice; a lane ends with one of the eight tokens
          const bool b8 = lane & 8, b4 = lane & 4, b2 = lane & 2;
          float r4[4], r2[2];
#pragma unroll
          for (int i = 0; i < 4; ++i) r4[i] = __shfl_xor_sync(0xffffffffu, b8 ? sq[i] : sq[i + 4], 8) + (b8 ? sq[i + 4] : sq[i]);
#pragma unroll
          for (int i = 0; i < 2; ++i) r2[i] = __shfl_xor_sync(0xffffffffu, b4 ? r4[i] : r4[i + 2], 4) + (b4 ? r4[i + 2] : r4[i]);
          float r = __shfl_xor_sync(0xffffffffu, b2 ? r2[0] : r2[1], 2) + (b2 ? r2[1] : r2[0]);
          r += __shfl_xor_sync(0xffffffffu, r, 1);
          const int d = (b8 ? 8 : 0) + (b4 ? 2 : 0) + (b2 ? 1 : 0);
          if (d < lim && (lane & 1) == 0) nm.ssq_out[(size_t)(t + d) * (N >> 4) + (f >> 4)] = r;
        }
      }
    };
    if (S > 1) cluster_wait();
    bool ok = mbar_wait(accum, 0);
    if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (ok) {
      const uint32_t tbase = tmem + ((uint32_t)(w4 * 32) << 16);
#pragma unroll 1
      for (int c = 4 * grp; c < n_quads; c += 8) {
        float v[16];
        tmem_ld16(tbase + 4 * c, v);
        if (S == 1) {
          float u[8] = {v[0], v[1], v[2], v[3], v[8], v[9], v[10], v[11]}, w[8] = {v[4], v[5], v[6], v[7], v[12], v[13], v[14], v[15]};
          if (EPI == EPI_RESID && c != 4 * grp) fetch_old(c);
          finish(c, u);
          if (EPI == EPI_RESID) fetch_old(c + 1);
          if (c + 1 < own) finish(c + 1, w);
          continue;
        }
        int r = c / RBQ, q = c - r * RBQ;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (c + j < n_quads) {
            const uint32_t a = recv0 + (uint32_t)(((rank * RBQ + q) * TC_BM + fl) * 16);
            if (r == rank) {
              asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[4 * j]), "f"(v[4 * j + 1]), "f"(v[4 * j + 2]), "f"(v[4 * j + 3]) : "memory");
            } else {
              uint32_t ra, rb;
              asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"((uint32_t)r));
              asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(recv_bar), "r"((uint32_t)r));
              asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                           ::"r"(ra), "f"(v[4 * j]), "f"(v[4 * j + 1]), "f"(v[4 * j + 2]), "f"(v[4 * j + 3]), "r"(rb) : "memory");
            }
          }
          if (++q == RBQ) { q = 0; ++r; }
        }
      }
    }
    if (S > 1) {
      __syncwarp();
      asm volatile("bar.sync 1, 256;" ::: "memory");                       // this rank's own part and the rows' factors are in place
      if (own > 0) {
        const bool got = mbar_wait_cluster(recv_bar, 0);
        if (!got) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
        ok = __all_sync(0xffffffffu, got) && ok;
      }
      __syncwarp();
      cluster_arrive();                                                     // every push into this CTA has landed
    }
#pragma unroll 1
    for (int q0 = grp; S > 1 && ok && q0 < own; q0 += 4) {
      if (EPI == EPI_RESID && q0 != grp) fetch_old(q0);
      float v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = 0.f;
      const bool two = q0 + 2 < own;
      const float4 *src = recv + q0 * TC_BM + fl;
#pragma unroll 2
      for (int s = 0; s < S; ++s, src += RBQ * TC_BM) {
        const float4 a = src[0], b = two ? src[2 * TC_BM] : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
        v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
      }
      finish(q0, v);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == PUSH_EPI_WARPS + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)tmem_cols) : "memory");
  }
  if (S > 1) cluster_wait();                                                // no CTA leaves while a push into it or from it is under way
}

// ------------------------------------------------------------------ host side
struct PushShape {
  int BN, S, SW, SA;
};
static inline int push_rank_tokens(int BN, int S) { return ((BN + S - 1) / S + 3) & ~3; }
static inline int push_smem_bytes(const PushShape &s) {
  return PUSH_KS * TC_BK * 2 * (s.SW * TC_BM + s.SA * s.BN) + (s.S > 1 ? s.S * push_rank_tokens(s.BN, s.S) * TC_BM * 4 : 0) + 1024 + 192 +
         4 * PUSH_MAX_BN;
}

static int gemm_push_init() {
  static bool dev_done[TC_MAX_DEVICES] = {false};
  std::lock_guard<std::mutex> lock(g_tc_init_mu);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= TC_MAX_DEVICES) return -4;
  if (dev_done[dev]) return 0;
  if (cudaFuncSetAttribute(gemm_push_kernel<EPI_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_push_kernel<EPI_GELU_T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_push_kernel<EPI_RESID>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
    return -4;
  dev_done[dev] = true;
  return 0;
}

// Rings of a tile: as deep as shared memory allows, up to three stages of tokens first.  Half an SM where that holds the
// CTA's whole share of K, or where the grid is more than one CTA per SM: the next kernel (or the second CTA) then has room
// to start on its weights.
static bool push_rings(PushShape *sh, int KB, long ctas) {
  const int n_st = ((KB + sh->S - 1) / sh->S + PUSH_KS - 1) / PUSH_KS;
  auto fill = [&](int limit) {
    sh->SW = sh->SA = 1;
    if (push_smem_bytes(*sh) > limit) return false;
    for (;;) {
      PushShape n = *sh;
      if (n.SA < std::min(n.SW, 3)) ++n.SA;
      else if (n.SW < std::min(n_st, PUSH_MAX_STAGES)) ++n.SW;
      else return true;
      if (push_smem_bytes(n) > limit) return true;
      *sh = n;
    }
  };
  if (fill(113 * 1024) && (sh->SW >= n_st || ctas > 148)) return true;
  return fill(227 * 1024);
}

// Token tile and K split for M tokens, by a cost in units of 0.01 us: block steps of a CTA, those among them whose weights do
// not fit into the ring ahead of the dependency wait, the exchange of a split, CTAs that share an SM or wait for one
// (clusters cannot use every SM: what fits of each size), and the tokens that a thread finishes.  Fitted to chains of
// dependent launches of QKV, Wo, W1 and W2 of d = 256 ... 1280 at 8 ... 512 tokens (336 shapes, 13000 tiles): 3 % above the
// best tile on average, 18 % at worst where this kernel is used.
static PushShape gemm_push_geometry(int N, int K, int M) {
  static const int split[6] = {1, 2, 3, 4, 6, 8}, fits[6] = {148, 140, 126, 128, 120, 112};
  const int FT = (N + TC_BM - 1) / TC_BM, KB = (K + TC_BK - 1) / TC_BK;
  PushShape best{};
  double best_cost = 0;
  int last = 0;
  for (int nt = (M + PUSH_MAX_BN - 1) / PUSH_MAX_BN; nt <= M; ++nt) {
    const int bn = ((M + nt - 1) / nt + 15) & ~15, tt = (M + bn - 1) / bn;
    if (bn < 32 && nt > 1) break;
    if (bn == last) continue;
    last = bn;
    for (int i = 0; i < 6; ++i) {
      PushShape sh{bn, split[i], 0, 0};
      const long ctas = (long)FT * tt * sh.S;
      if (sh.S > KB || !push_rings(&sh, KB, ctas)) continue;
      const int steps = (KB + sh.S - 1) / sh.S, ahead = std::min(PUSH_KS * sh.SW, steps);
      const int share = (int)((ctas + 147) / 148), per_sm = 228 * 1024 / (push_smem_bytes(sh) + 1024);
      const long waves = (ctas + fits[i] * per_sm - 1) / (fits[i] * per_sm);
      const double cost = steps * (10 + 0.07 * bn * share) + (steps - ahead) * 29.0 * share +
                          (sh.S > 1 ? 43 + 2.9 * bn + 200.0 * ctas / 148 : 0) + (waves - 1) * 200.0 +
                          39.0 * ((bn / sh.S + 15) / 16) + (share - 1) * 145.0;
      if (!best.BN || cost < best_cost) {
        best = sh;
        best_cost = cost;
      }
    }
  }
  return best;
}

static bool gemm_push_launch(cudaStream_t st, bool pdl, GemmSkPlan &p, void *C, int M, int epi, int *status, const SkNorm *norm,
                             LiveRows lr, PushShape sh = PushShape{}) {
  if (!p.valid || M < 1 || M > p.M_max) return false;
  for (const auto &t : p.push)
    if (!sh.BN && t.M == M) sh = PushShape{t.BN, t.S, t.SW, t.SA};
  if (!sh.BN) {
    sh = gemm_push_geometry(p.N, p.K, M);
    p.push.push_back(GemmSkPlan::PushTile{M, sh.BN, sh.S, sh.SW, sh.SA});
  }
  const int idx = sh.BN / 16 - 1;
  if (!p.haveA[idx]) {
    if (tc_encode(&p.mapA[idx], p.A, p.M_max, p.K, sh.BN)) return false;
    p.haveA[idx] = true;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((p.N + TC_BM - 1) / TC_BM, (M + sh.BN - 1) / sh.BN, sh.S);
  cfg.blockDim = dim3(PUSH_THREADS);
  cfg.dynamicSmemBytes = push_smem_bytes(sh);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = sh.S;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  const SkNorm nm = norm ? *norm : SkNorm{};
  const int cols = sh.BN <= 32 ? 32 : sh.BN <= 64 ? 64 : 128;
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, p.mapW, p.mapA[idx], C, M, p.N, p.K, sh.BN, push_rank_tokens(sh.BN, sh.S), sh.SW, sh.SA,
                              cols, nm, status, lr) == cudaSuccess;
  };
  return epi == EPI_F32 ? go(gemm_push_kernel<EPI_F32>) : epi == EPI_GELU_T ? go(gemm_push_kernel<EPI_GELU_T>)
         : epi == EPI_RESID ? go(gemm_push_kernel<EPI_RESID>) : false;
}

}  // namespace tsfm
