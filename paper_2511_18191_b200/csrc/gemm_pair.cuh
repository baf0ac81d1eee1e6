// bf16 x bf16 -> fp32 contraction of many tokens on pairs of SMs (tcgen05, cta_group::2).
//
//   C[t, f] (op)= sum_k A[t, k] * W[f, k]        A: [M, K] tokens, W: [N, K] weights
//
// Bound: an SM's shared memory fills from L2 at 64 bytes per cycle, and a 128 x 128 x 64 block step needs
// 32 KB (512 cycles) for 260 cycles of tensor work.  Two SMs that work on one tile of 256 features x BN
// tokens each load their half of both operands (128 feature rows, BN / 2 token rows) and both halves feed
// both tensor cores: 256 + BN cycles of fill for 2 BN cycles of work per block step and SM, i.e. balanced
// at BN = 256 where the single-SM form needs 2.5 times the work's time.
//   * cluster of 2 along x; rank r owns features 128 r ... 128 r + 127 of the pair's tile in its own
//     tensor memory, rank 0 issues every MMA; the copies of both ranks report to rank 0's barriers, the
//     commits arrive at both ranks' (no copy is multicast);
//   * persistent: pairs walk the tiles; with two accumulators (2 BN <= 512 columns) the epilogue of a tile
//     runs under the main loop of the next;
//   * 8 epilogue warps in two groups take 32-token chunks in turn: tcgen05.ld, conversion, staged as
//     [token][128 features] and written (fp32, bf16, GELU -> bf16) or added to x by the TMA unit.
// Warps 0-7 epilogue, 8 TMA producer, 9 tensor-memory allocation and MMA issue.  Waits are bounded as in
// gemm_tc.cuh.
#pragma once
#include "gemm_sk.cuh"

namespace tsfm {

constexpr int PAIR_CHUNK = 32;                   // tokens per epilogue chunk
constexpr int PAIR_THREADS = 320;
constexpr int PAIR_MAX = 74;                     // pairs of SMs on the device
constexpr int PAIR_STAGE_OUT = PAIR_CHUNK * TC_BM * 4;   // staging per epilogue group

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// Copy whose bytes are reported to the even rank's barrier at the same offset (bit 24 of a shared::cluster
// address tells the two ranks of a pair apart).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar & 0xFEFFFFFFu) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
// Arrives at the barrier of this offset in both ranks once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void mbar_arrive_rank0(uint32_t bar) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(bar), "r"(0u));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
// Bounded wait that also acquires what the other rank released.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if (it == 256) t0 = globaltimer_ns();
    if (it > 256 && (it & 255) == 0 && globaltimer_ns() - t0 > TC_WAIT_NS) return false;
  }
}
// 32 consecutive columns of this thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// grid = 2 x pairs, cluster = 2.  C leaves through mapC (box 128 features x 32 tokens): tma_c = SK_TMA_F32 /
// SK_TMA_BF16 (stores; epi tells GELU) or SK_TMA_ADD.
__global__ void __launch_bounds__(PAIR_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapA,
                 const __grid_constant__ CUtensorMap mapC, int M, int N, int K, int BN, int stages, int n_acc,
                 int tmem_cols, int epi, int tma_c, int *__restrict__ status, const LiveRows lr) {
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (lr.n_live) M = min(M, *reinterpret_cast<const volatile int *>(lr.n_live) * lr.q_len);
  const int FT = (N + 2 * TC_BM - 1) / (2 * TC_BM), n_tiles = FT * ((M + BN - 1) / BN);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const uint32_t rank = blockIdx.x & 1;                        // == %cluster_ctarank
  if (pair >= n_tiles) return;                                 // both ranks alike
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int a_bytes = (BN / 2) * TC_BK * 2, stage_bytes = TC_W_BYTES + a_bytes;
  const uint32_t out0 = tiles + (uint32_t)(stages * stage_bytes);
  const uint32_t bars = out0 + 2 * PAIR_STAGE_OUT;
  const uint32_t full0 = bars, empty0 = bars + 64, acc_full0 = bars + 128, acc_empty0 = bars + 144, slot = bars + 160;
  uint32_t *slot_ptr = reinterpret_cast<uint32_t *>(smem_raw + (slot - smem_u32(smem_raw)));
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int KB = (K + TC_BK - 1) / TC_BK;

  if (warp == 8 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapW) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapC) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(acc_full0 + 8 * s, 1);
      mbar_init(acc_empty0 + 8 * s, 16);                       // 8 epilogue warps of each rank
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"((uint32_t)tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                          // both ranks' barriers stand before any copy reports to them
  tc_fence_after();
  const uint32_t tmem = *slot_ptr;

  if (warp == 8) {
    if (elect_one()) {
      // ---------------- TMA producer: this rank's half of both operands.  The first ring-full of weight
      // tiles is requested before the dependency wait.
      const int total = ((n_tiles - pair + n_pairs - 1) / n_pairs) * KB;   // block steps of all tiles of this pair
      const int pre = total < stages ? total : stages;
      // position of the next copy (the divisions of a tile switch stay out of the block steps)
      struct Pos {
        int tile, kb, wy, ay;
      };
      auto at_tile = [&](Pos &p, int tile) {
        p.tile = tile;
        p.kb = 0;
        p.wy = (tile % FT) * 2 * TC_BM + (int)rank * TC_BM;
        p.ay = (tile / FT) * BN + (int)rank * (BN / 2);
      };
      auto next = [&](Pos &p) {
        if (++p.kb == KB) at_tile(p, p.tile + n_pairs);
      };
      Pos pw, pa;
      at_tile(pw, pair);
      pa = pw;
      uint32_t dst = tiles, bar = full0;
      for (int it = 0; it < pre; ++it, dst += stage_bytes, bar += 8, next(pw)) {
        if (rank == 0) mbar_expect_tx(bar, 2u * (uint32_t)stage_bytes);
        tma_load_2d_pair(dst, &mapW, pw.kb * TC_BK, pw.wy, bar);
      }
      pdl_sync();
      dst = tiles, bar = full0;
      for (int it = 0; it < pre; ++it, dst += stage_bytes, bar += 8, next(pa))
        tma_load_2d_pair(dst + TC_W_BYTES, &mapA, pa.kb * TC_BK, pa.ay, bar);
      int s = 0;
      uint32_t ph = 0;
      dst = tiles;
      for (int it = pre; it < total; ++it, next(pa)) {
        if (!mbar_wait_cluster(empty0 + 8 * s, ph)) { atomicExch(status, DEV_TIMEOUT_TMA); break; }
        if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2u * (uint32_t)stage_bytes);
        tma_load_2d_pair(dst, &mapW, pa.kb * TC_BK, pa.wy, full0 + 8 * s);
        tma_load_2d_pair(dst + TC_W_BYTES, &mapA, pa.kb * TC_BK, pa.ay, full0 + 8 * s);
        dst += stage_bytes;
        if (++s == stages) { s = 0; ph ^= 1u; dst = tiles; }
      }
    }
  } else if (warp == 9) {
    if (rank == 0 && elect_one()) {
      // ---------------- MMA issuer
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(2 * TC_BM >> 4) << 24);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int tile = pair, i = 0; tile < n_tiles && ok; tile += n_pairs, ++i) {
        const int buf = n_acc == 2 ? (i & 1) : 0, use = n_acc == 2 ? (i >> 1) : i;
        if (!mbar_wait_cluster(acc_empty0 + 8 * buf, ((uint32_t)use & 1u) ^ 1u)) { atomicExch(status, DEV_TIMEOUT_MMA); break; }
        tc_fence_after();
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait_cluster(full0 + 8 * s, ph)) { atomicExch(status, DEV_TIMEOUT_MMA); ok = false; break; }
          tc_fence_after();
          const uint32_t sw = tiles + s * stage_bytes;
          const uint64_t dw = umma_smem_desc(sw), da = umma_smem_desc(sw + TC_W_BYTES);
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            umma_bf16_pair(tmem + (uint32_t)(buf * BN), dw + 2 * k, da + 2 * k, idesc, (kb | k) ? 1u : 0u);
          umma_commit_pair(empty0 + 8 * s);
          if (++s == stages) { s = 0; ph ^= 1u; }
        }
        if (ok) umma_commit_pair(acc_full0 + 8 * buf);
      }
    }
  } else {
    // ---------------- epilogue
    const int grp = warp >> 2, w4 = warp & 3, fl = w4 * 32 + lane;
    const uint32_t stage = out0 + (uint32_t)(grp * PAIR_STAGE_OUT);
    float *stage_f = reinterpret_cast<float *>(smem_raw + (stage - smem_u32(smem_raw)));
    bf16 *stage_h = reinterpret_cast<bf16 *>(stage_f);
    const bool leader = (threadIdx.x & 127) == 0;
    pdl_sync();
    bool ok = true;
    for (int tile = pair, i = 0; tile < n_tiles; tile += n_pairs, ++i) {
      const int buf = n_acc == 2 ? (i & 1) : 0, use = n_acc == 2 ? (i >> 1) : i;
      const int f0 = (tile % FT) * 2 * TC_BM + (int)rank * TC_BM, t0 = (tile / FT) * BN;
      if (ok) {                                                // (after a wait that ran out: no more waits, nothing stored)
        ok = mbar_wait_cluster(acc_full0 + 8 * buf, (uint32_t)use & 1u);
        if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
      }
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(w4 * 32) << 16) + (uint32_t)(buf * BN);
      for (int c = grp * PAIR_CHUNK; c < BN; c += 2 * PAIR_CHUNK) {
        if (t0 + c >= M) break;
        float v[PAIR_CHUNK];
        tmem_ld32(tbase + c, v);
        // the staging tile is free once its previous copy has been read
        if (leader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        if (tma_c == SK_TMA_BF16) {
          if (epi == EPI_GELU_T) {
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; ++j) stage_h[j * TC_BM + fl] = __float2bfloat16_rn(gelu_erf_fast(v[j]));
          } else {
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; ++j) stage_h[j * TC_BM + fl] = __float2bfloat16_rn(v[j]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; ++j) stage_f[j * TC_BM + fl] = v[j];
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        if (leader && ok && f0 < N) {
          if (tma_c == SK_TMA_ADD)
            asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(&mapC), "r"(f0), "r"(t0 + c), "r"(stage) : "memory");
          else
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(&mapC), "r"(f0), "r"(t0 + c), "r"(stage) : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      // accumulator drained: rank 0 may overwrite it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_rank0(acc_empty0 + 8 * buf);
    }
    if (leader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();          // no rank leaves while the other's MMAs read its shared memory or its arrivals are under way
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------ host side
struct PairShape {
  int BN, stages, n_acc, tmem_cols, pairs, smem_bytes;
};

static int gemm_pair_init() {
  static bool dev_done[TC_MAX_DEVICES] = {false};
  std::lock_guard<std::mutex> lock(g_tc_init_mu);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= TC_MAX_DEVICES) return -4;
  if (dev_done[dev]) return 0;
  if (cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) return -4;
  dev_done[dev] = true;
  return 0;
}

// Tile rule: see the header for the cost of a block step; the epilogue of a pair's last tile is not hidden.
static PairShape gemm_pair_geometry(int N, int K, int M) {
  const int FT = (N + 2 * TC_BM - 1) / (2 * TC_BM), KB = (K + TC_BK - 1) / TC_BK;
  PairShape sh{};
  long best = 0;
  for (int bn = 32; bn <= 256; bn += 32) {
    const int tiles = FT * ((M + bn - 1) / bn);
    const long waves = (tiles + PAIR_MAX - 1) / PAIR_MAX;
    const long cost = waves * KB * (256 + (bn < 96 ? 96 : bn)) + 8 * bn + 20 * (tiles < PAIR_MAX ? tiles : PAIR_MAX);
    if (!best || cost < best) {
      best = cost;
      sh.BN = bn;
    }
  }
  return sh;
}
// Shapes and outputs it takes: whole 128-feature tiles leave through the TMA unit.
static bool gemm_pair_eligible(const GemmSkPlan &p, const void *C) { return p.valid && p.N % TC_BM == 0 && !((uintptr_t)C & 15); }

// Ring depth and tensor memory of a tile width for M tokens.
static void gemm_pair_fill(PairShape *sh, int N, int K, int M) {
  const int FT = (N + 2 * TC_BM - 1) / (2 * TC_BM);
  const int tiles = FT * ((M + sh->BN - 1) / sh->BN);
  sh->pairs = tiles < PAIR_MAX ? tiles : PAIR_MAX;
  sh->n_acc = tiles > PAIR_MAX ? 2 : 1;
  const int cols = sh->BN * sh->n_acc;
  sh->tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
  const int stage = TC_W_BYTES + sh->BN / 2 * TC_BK * 2;
  const int st = (227 * 1024 - 2 * PAIR_STAGE_OUT - 2048) / stage;
  if (sh->stages == 0) sh->stages = st > 8 ? 8 : st;
  sh->smem_bytes = sh->stages * stage + 2 * PAIR_STAGE_OUT + 1024 + 256;
}

static bool gemm_pair_launch(cudaStream_t st, bool pdl, GemmSkPlan &p, void *C, int M, int epi, int *status, LiveRows lr,
                             PairShape sh = PairShape{}) {
  if (M < 1 || M > p.M_max) return false;
  if (!sh.BN) {
    sh = gemm_pair_geometry(p.N, p.K, M);
    gemm_pair_fill(&sh, p.N, p.K, M);
  }
  const int idx = sh.BN / 32 - 1;
  if (!p.haveA2[idx]) {
    if (tc_encode(&p.mapA2[idx], p.A, p.M_max, p.K, sh.BN / 2)) return false;
    p.haveA2[idx] = true;
  }
  const int tma_c = epi == EPI_RESID ? SK_TMA_ADD : epi == EPI_F32 ? SK_TMA_F32 : SK_TMA_BF16;
  const CUtensorMap *mapC = sk_map_c(p, C, M, PAIR_CHUNK, tma_c == SK_TMA_BF16);
  if (!mapC) return false;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * sh.pairs);
  cfg.blockDim = dim3(PAIR_THREADS);
  cfg.dynamicSmemBytes = sh.smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel, p.mapW, p.mapA2[idx], *mapC, M, p.N, p.K, sh.BN, sh.stages, sh.n_acc,
                            sh.tmem_cols, epi, tma_c, status, lr) == cudaSuccess;
}

}  // namespace tsfm
