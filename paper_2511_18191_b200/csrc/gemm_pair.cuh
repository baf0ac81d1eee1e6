// bf16 x bf16 -> fp32 contraction of many tokens on pairs of SMs (tcgen05, cta_group::2).
//
//   C[t, f] (op)= sum_k A[t, k] * W[f, k]        A: [M, K] tokens, W: [N, K] weights
//
// Bound: an SM's shared memory fills from L2 at 64 bytes per cycle, and a 128 x 128 x 64 block step needs
// 32 KB (512 cycles) for 260 cycles of tensor work.  Two SMs that work on one tile of 256 features x BN
// tokens each load their half of both operands (128 feature rows, BN / 2 token rows) and both halves feed
// both tensor cores: 256 + BN cycles of fill for 2 BN cycles of work per block step and SM, i.e. balanced
// at BN = 256 where the single-SM form needs twice the work's time.
//   * cluster of 2 along x (4 where two pairs share a tile, each with half of K); rank r owns features
//     128 r ... 128 r + 127 of the pair's tile in its own tensor memory, rank 0 issues every MMA; the copies of
//     both ranks report to rank 0's barriers, the commits arrive at both ranks' (no copy is multicast);
//   * persistent: pairs walk the tiles; with two accumulators (2 BN <= 512 columns) the epilogue of a tile
//     runs under the main loop of the next;
//   * 16 epilogue warps in four groups.  Where a pair walks over several tiles they take 16-token chunks in turn: tcgen05.ld,
//     conversion, staged as [token][128 features] and written (fp32, bf16, GELU -> bf16) or added to x by the TMA unit, all of
//     it under the next tile's main loop.  Where every pair has one tile nothing hides the epilogue, and plain fp32 outputs (QKV
//     of short passes) leave straight from registers, eight rows of a feature per lane: 0.6 to 1.4 us less at 576 to 1280 tokens
//     of d = 768 ... 1280 (GELU that way between 0.7 us less and 1.1 more, residual updates up to 0.7 more: their stores share
//     the issue slots with the conversions);
//   * the MMA warp runs its loop as a whole and one lane issues (see gemm_push_kernel): 0.1 to 0.5 us a contraction;
//   * RMSNorms can be folded in (SkNorm; slices of 128 features): a residual epilogue fetches the old rows
//     while the main loop runs, and emits x, the next operand bf16(gain x) and the rows' sums of squares; a
//     consumer scales its rows.  Used where an RMSNorm launch costs more than that (kPairFoldMaxRows);
//   * the QKV contraction of a pass of several query tiles rotates its queries and keys and puts keys and
//     values into the cache as bf16 (PairRope): 43 us instead of 34 + 14 (kv_append_kernel) at 6000 x 1024,
//     142 instead of 132 + 47 at 16320 x 1280.
// Graph replay of dependent launches, gemm_sk_kernel -> this one: M = 16320, d = 1280: QKV 158 -> 118 us
// (1355 TFLOP/s), W1 with GELU 254 -> 160, W2 175 -> 149, Wo 67 -> 50; M = 6000, d = 1024: 47 -> 34, 74 -> 40,
// 61 -> 44, 21 -> 16.
// Warps 0-15 epilogue, 16 TMA producer, 17 tensor-memory allocation and MMA issue, 18-19 the rows' factors and
// cache positions of the next tile.  (With 8 epilogue warps the folded forms, a chain of latencies per chunk, set
// the pace: QKV of 6000 x 1024 60 us.)  Waits are bounded as in gemm_tc.cuh.
#pragma once
#include "gemm_sk.cuh"

namespace tsfm {

// How an output leaves: from registers (fp32), or through the TMA unit: fp32 added to what is there, bf16 stored, fp32 stored.
enum { SK_TMA_NONE = 0, SK_TMA_ADD = 1, SK_TMA_BF16 = 2, SK_TMA_F32 = 3 };
constexpr int PAIR_CHUNK = 16;                   // tokens per epilogue chunk
constexpr int PAIR_GROUPS = 4, PAIR_EPI_WARPS = 4 * PAIR_GROUPS, PAIR_ROW_WARPS = 2;
constexpr int PAIR_THREADS = 32 * (PAIR_EPI_WARPS + 2 + PAIR_ROW_WARPS);
constexpr int PAIR_MAX_STAGES = 8;
constexpr int PAIR_MAX = 74;                     // pairs of SMs on the device
constexpr int PAIR_STAGE_OUT = PAIR_CHUNK * TC_BM * 4;   // staging per epilogue group
constexpr int PAIR_ROW_BYTES = 2 * 256 * (4 + 8);        // factors and cache positions of two tiles' rows

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
// Arrives at the barrier of this offset in both ranks of a pair (mask) once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint32_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)mask) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_rank(uint32_t bar, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(bar), "r"(rank));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
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
// Rotary positions and cache append of a QKV contraction (N = 3 d, d % 128 == 0): features [0, d) become
// rotated queries, scaled for base-2 softmax, fp32 in C; [d, 2 d) rotated keys and [2 d, 3 d) values go to the
// cache only.
struct PairRope {
  const float2 *rope;              // [cap][dh / 2], NULL: an ordinary contraction
  bf16 *Kc, *Vc;                   // this layer's cache [B][heads][cap][dh]
  PassGeom g;
  int n_heads, dh;
};

// Four rows of a staged chunk (one warp): queries and keys rotated, queries to C, keys and values to the cache.
// A lane takes both members of two rotation pairs; cs holds their table entries, fetched a chunk ahead (a round
// trip to L2 per chunk otherwise).
struct PairRopeLane {
  int dim, hl, lph;                // first of the lane's two dims below dh / 2; first feature of its head in the tile
  __device__ __forceinline__ PairRopeLane(int lane, int dh) {
    lph = dh >> 2;
    dim = (lane & (lph - 1)) * 2;
    hl = (lane / lph) * dh;
  }
};
__device__ __forceinline__ void pair_rope_fetch(float4 (&cs)[PAIR_CHUNK / 4], const int2 *pos, int w4, int t0, int M, int half, int dim,
                                                const float2 *rope) {
#pragma unroll
  for (int r = 0; r < PAIR_CHUNK / 4; ++r) {
    const int tl = w4 * (PAIR_CHUNK / 4) + r;
    cs[r] = make_float4(1.f, 0.f, 1.f, 0.f);
    if (t0 + tl < M) cs[r] = *reinterpret_cast<const float4 *>(rope + (size_t)pos[tl].y * half + dim);   // cos sin cos sin
  }
}
__device__ __forceinline__ void pair_rope_rows(const float *stage, const int2 *pos, const float4 (&cs)[PAIR_CHUNK / 4], int w4,
                                               const PairRopeLane &pl, int f0, int t0, int M, int N, float *C, const PairRope &pr) {
  const int d = N / 3, part = f0 / d, dh = pr.dh, half = dh >> 1;
  const int head = (f0 - part * d + pl.hl) / dh;
  const float sc = rsqrtf((float)dh) * 1.4426950408889634f;
#pragma unroll
  for (int r = 0; r < PAIR_CHUNK / 4; ++r) {
    const int tl = w4 * (PAIR_CHUNK / 4) + r, t = t0 + tl;
    if (t >= M) break;
    const float2 u = *reinterpret_cast<const float2 *>(stage + tl * TC_BM + pl.hl + pl.dim);
    const float2 y = *reinterpret_cast<const float2 *>(stage + tl * TC_BM + pl.hl + pl.dim + half);
    const float2 a = make_float2(u.x * cs[r].x - y.x * cs[r].y, u.y * cs[r].z - y.y * cs[r].w);
    const float2 b = make_float2(y.x * cs[r].x + u.x * cs[r].y, y.y * cs[r].z + u.y * cs[r].w);
    if (part == 0) {
      float *dst = C + (size_t)t * N + f0 + pl.hl + pl.dim;
      *reinterpret_cast<float2 *>(dst) = make_float2(a.x * sc, a.y * sc);
      *reinterpret_cast<float2 *>(dst + half) = make_float2(b.x * sc, b.y * sc);
    } else {
      const int2 bp = pos[tl];
      bf16 *dst = (part == 1 ? pr.Kc : pr.Vc) + (((size_t)bp.x * pr.n_heads + head) * pr.g.cap + bp.y) * dh + pl.dim;
      *reinterpret_cast<uint32_t *>(dst) = part == 1 ? pack_bf16x2(a.x, a.y) : pack_bf16x2(u.x, u.y);
      *reinterpret_cast<uint32_t *>(dst + half) = part == 1 ? pack_bf16x2(b.x, b.y) : pack_bf16x2(y.x, y.y);
    }
  }
}

// grid = 2 x split x pairs, cluster = 2 x split (split: pairs per tile).  C leaves through mapC (box 128 features x 16 tokens): tma_c = SK_TMA_F32 /
// SK_TMA_BF16 (stores; epi tells GELU) or SK_TMA_ADD; SK_TMA_NONE: fp32, straight from registers.
__global__ void __launch_bounds__(PAIR_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapA,
                 const __grid_constant__ CUtensorMap mapC, int M, int N, int K, int BN, int split, int stages, int n_acc,
                 int tmem_cols, int epi, int tma_c, float *C, const SkNorm nm, const PairRope pr, int *__restrict__ status,
                 const LiveRows lr) {
  // rows in use (active-series compaction): read before the dependency wait, see gemm_sk_kernel
  if (lr.n_live) M = min(M, *reinterpret_cast<const volatile int *>(lr.n_live) * lr.q_len);
  const int FT = (N + 2 * TC_BM - 1) / (2 * TC_BM), n_tiles = FT * ((M + BN - 1) / BN);
  // rank within the pair; which half of K the pair takes (split == 2: two pairs, a cluster of four, on one tile)
  const uint32_t rank = blockIdx.x & 1, half = split == 2 ? (blockIdx.x >> 1) & 1 : 0;
  const int pair = blockIdx.x / (2 * split), n_pairs = gridDim.x / (2 * split);
  if (pair >= n_tiles) return;                                 // the whole cluster alike
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int a_bytes = (BN / 2) * TC_BK * 2, stage_bytes = TC_W_BYTES + a_bytes;
  const uint32_t out0 = tiles + (uint32_t)(stages * stage_bytes);
  const uint32_t bars = out0 + PAIR_GROUPS * PAIR_STAGE_OUT;
  const uint32_t full0 = bars, empty0 = bars + 64, acc_full0 = bars + 128, acc_empty0 = bars + 144, slot = bars + 160;
  const uint32_t rows_full0 = bars + 176, rows_empty0 = bars + 192, recv_bar = bars + 208;
  const uint32_t recv0 = bars + 256 + PAIR_ROW_BYTES;          // (split) the other pair's sums of the rows finished here: [quad][feature] x 4 rows
  float *row_scale = reinterpret_cast<float *>(smem_raw + (bars + 256 - smem_u32(smem_raw)));   // [2 tiles][256]
  int2 *row_pos = reinterpret_cast<int2 *>(row_scale + 512);                                    // [2 tiles][256] (series, position)
  uint32_t *slot_ptr = reinterpret_cast<uint32_t *>(smem_raw + (slot - smem_u32(smem_raw)));
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int KB_all = (K + TC_BK - 1) / TC_BK, kb0 = KB_all * (int)half / split, KB = KB_all * ((int)half + 1) / split - kb0;
  // rows of the tile that this pair finishes
  const int r_beg = (int)half * (BN / split), r_end = r_beg + BN / split;

  if (warp == PAIR_EPI_WARPS && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapW) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapC) : "memory");
  }
  if (warp == 0) {
    if (lane < PAIR_MAX_STAGES) {
      mbar_init(full0 + 8 * lane, 1);
      mbar_init(empty0 + 8 * lane, 1);
    }
    if (lane < 2) {
      mbar_init(acc_full0 + 8 * lane, 1);
      mbar_init(acc_empty0 + 8 * lane, 2 * PAIR_EPI_WARPS);    // of both ranks
      mbar_init(rows_full0 + 8 * lane, PAIR_ROW_WARPS);
      mbar_init(rows_empty0 + 8 * lane, PAIR_EPI_WARPS);
    }
    if (lane == 0 && split == 2) {
      mbar_init(recv_bar, 1);
      const int rows = min(M - (pair / FT) * BN, r_end) - r_beg;             // in whole chunks
      mbar_expect_tx(recv_bar, rows > 0 ? (uint32_t)((rows + PAIR_CHUNK - 1) / PAIR_CHUNK * PAIR_STAGE_OUT) : 0u);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
  }
  if (warp == PAIR_EPI_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"((uint32_t)tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                          // both ranks' barriers stand before any copy reports to them
  tc_fence_after();
  const uint32_t tmem = *slot_ptr;

  if (warp == PAIR_EPI_WARPS) {
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
        tma_load_2d_pair(dst, &mapW, (kb0 + pw.kb) * TC_BK, pw.wy, bar);
      }
      pdl_sync();
      dst = tiles, bar = full0;
      for (int it = 0; it < pre; ++it, dst += stage_bytes, bar += 8, next(pa))
        tma_load_2d_pair(dst + TC_W_BYTES, &mapA, (kb0 + pa.kb) * TC_BK, pa.ay, bar);
      int s = 0;
      uint32_t ph = 0;
      dst = tiles;
      for (int it = pre; it < total; ++it, next(pa)) {
        if (!mbar_wait_cluster(empty0 + 8 * s, ph)) { atomicExch(status, DEV_TIMEOUT_TMA); break; }
        if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2u * (uint32_t)stage_bytes);
        tma_load_2d_pair(dst, &mapW, (kb0 + pa.kb) * TC_BK, pa.wy, full0 + 8 * s);
        tma_load_2d_pair(dst + TC_W_BYTES, &mapA, (kb0 + pa.kb) * TC_BK, pa.ay, full0 + 8 * s);
        dst += stage_bytes;
        if (++s == stages) { s = 0; ph ^= 1u; dst = tiles; }
      }
    }
  } else if (warp == PAIR_EPI_WARPS + 1) {
    if (rank == 0) {
      // ---------------- MMA issuer
      const bool leader = elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(2 * TC_BM >> 4) << 24);
      pdl_sync();                                              // (the limit on the waits below starts with the input, not before)
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      const uint64_t dw0 = umma_smem_desc(tiles);
      uint64_t dw = dw0;
      for (int tile = pair, i = 0; tile < n_tiles && ok; tile += n_pairs, ++i) {
        const int buf = n_acc == 2 ? (i & 1) : 0, use = n_acc == 2 ? (i >> 1) : i;
        if (!mbar_wait_cluster(acc_empty0 + 8 * buf, ((uint32_t)use & 1u) ^ 1u)) { atomicExch(status, DEV_TIMEOUT_MMA); break; }
        tc_fence_after();
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait_cluster(full0 + 8 * s, ph)) { atomicExch(status, DEV_TIMEOUT_MMA); ok = false; break; }
          const uint64_t da = dw + (TC_W_BYTES >> 4);
          if (leader) {
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)
              umma_bf16_pair(tmem + (uint32_t)(buf * BN), dw + 2 * k, da + 2 * k, idesc, (kb | k) ? 1u : 0u);
            umma_commit_pair(empty0 + 8 * s, 3u << (2 * half));
          }
          dw += (uint32_t)(stage_bytes >> 4);
          if (++s == stages) { s = 0; ph ^= 1u; dw = dw0; }
        }
        if (ok && leader) umma_commit_pair(acc_full0 + 8 * buf, 3u << (2 * half));
      }
      __syncwarp();
    }
  } else if (warp >= PAIR_EPI_WARPS + 2) {
    // ---------------- factors (folded norm) and cache positions of the rows of each tile
    pdl_sync();
    if (nm.ssq_in || pr.rope) {
      for (int tile = pair, i = 0; tile < n_tiles; tile += n_pairs, ++i) {
        const int rb = i & 1, t0 = (tile / FT) * BN;
        const bool ok = mbar_wait(rows_empty0 + 8 * rb, ((uint32_t)(i >> 1) & 1u) ^ 1u);
        if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
        if (!__all_sync(0xffffffffu, ok)) break;
        for (int r = threadIdx.x - 32 * (PAIR_EPI_WARPS + 2); r < BN && t0 + r < M; r += 32 * PAIR_ROW_WARPS) {
          const int t = t0 + r;
          if (nm.ssq_in) {
            const float *src = nm.ssq_in + (size_t)t * nm.n_part;
            float acc = 0.f;
            for (int j0 = 0; j0 < nm.n_part; j0 += 16) {         // (one round trip up to d = 2048)
              float v[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] = j0 + j < nm.n_part ? __ldcg(src + j0 + j) : 0.f;
#pragma unroll
              for (int j = 0; j < 16; ++j) acc += v[j];
            }
            row_scale[rb * 256 + r] = rsqrtf(acc * nm.inv_d + nm.eps);
          }
          if (pr.rope) {
            const SlotPos sp = slot_lookup(pr.g, t / pr.g.q_len);
            row_pos[rb * 256 + r] = make_int2(sp.b, sp.p0 + t % pr.g.q_len);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(rows_full0 + 8 * rb);
      }
    }
  } else {
    // ---------------- epilogue
    const int grp = warp >> 2, w4 = warp & 3, fl = w4 * 32 + lane;
    const uint32_t stage = out0 + (uint32_t)(grp * PAIR_STAGE_OUT);
    float *stage_f = reinterpret_cast<float *>(smem_raw + (stage - smem_u32(smem_raw)));
    bf16 *stage_h = reinterpret_cast<bf16 *>(stage_f);
    uint16_t *stage_u = reinterpret_cast<uint16_t *>(stage_f);
    const bool leader = (threadIdx.x & 127) == 0;
    const PairRopeLane pl(lane, pr.rope ? pr.dh : 64);
    const bool direct = tma_c == SK_TMA_NONE && !pr.rope;
    const bool produce = nm.a_out != nullptr;                  // residual update with the next norm's operand
    pdl_sync();
    bool ok = true;
    for (int tile = pair, i = 0; tile < n_tiles; tile += n_pairs, ++i) {
      const int buf = n_acc == 2 ? (i & 1) : 0, use = n_acc == 2 ? (i >> 1) : i;
      const int f0 = (tile % FT) * 2 * TC_BM + (int)rank * TC_BM, t0 = (tile / FT) * BN;
      const int fc = f0 + lane * 4;                            // features this lane finishes in row order
      const float *scale = row_scale + (i & 1) * 256;
      const int2 *pos = row_pos + (i & 1) * 256;
      // old values of the group's first chunk: while the main loop runs
      float4 gain = make_float4(0.f, 0.f, 0.f, 0.f);
      float old[PAIR_CHUNK];
      auto fetch_old = [&](int c) {
#pragma unroll
        for (int j = 0; j < PAIR_CHUNK; ++j)
          old[j] = (c < r_end && t0 + c + j < M && f0 < N) ? __ldcg(C + (size_t)(t0 + c + j) * N + f0 + fl) : 0.f;
      };
      if (produce) {
        if (f0 < N) gain = *reinterpret_cast<const float4 *>(nm.gain + fc);
        fetch_old(r_beg + grp * PAIR_CHUNK);
      }
      // (after a wait that ran out: no more waits, nothing stored)
      if (ok && (nm.ssq_in || pr.rope)) ok = mbar_wait(rows_full0 + 8 * (i & 1), (uint32_t)(i >> 1) & 1u);
      float4 cs[PAIR_CHUNK / 4];
      const bool rotate = pr.rope && f0 < 2 * (N / 3);         // queries and keys
      if (ok && rotate) pair_rope_fetch(cs, pos + grp * PAIR_CHUNK, w4, t0 + grp * PAIR_CHUNK, grp * PAIR_CHUNK < BN ? M : 0, pr.dh >> 1, pl.dim, pr.rope);
      if (ok) ok = mbar_wait_cluster(acc_full0 + 8 * buf, (uint32_t)use & 1u);
      if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);       // (either wait)
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(w4 * 32) << 16) + (uint32_t)(buf * BN);
      if (direct) {
        // A lane holds a feature of eight rows: 128 bytes of a row per warp and store.
        for (int c = grp * (BN / PAIR_GROUPS), end = c + BN / PAIR_GROUPS; c < end && t0 + c < M; c += 8) {
          float v[8];
          tmem_ld8(tbase + c, v);
          if (nm.ssq_in) {
            const float4 k0 = *reinterpret_cast<const float4 *>(scale + c), k1 = *reinterpret_cast<const float4 *>(scale + c + 4);
            v[0] *= k0.x; v[1] *= k0.y; v[2] *= k0.z; v[3] *= k0.w;
            v[4] *= k1.x; v[5] *= k1.y; v[6] *= k1.z; v[7] *= k1.w;
          }
          const int lim = ok && f0 < N ? M - t0 - c : 0;
          float *dst = C + (size_t)(t0 + c) * N + f0 + fl;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (j < lim) dst[(size_t)j * N] = v[j];
        }
      }
      if (split == 2) {
        // the sums of the rows that the other pair finishes go to the CTA with the same features there (see gemm_push_kernel)
        const int o_beg = BN / 2 - r_beg;                      // (0 or BN / 2)
        uint32_t there, bar_there;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(recv0 + (uint32_t)fl * 16), "r"((blockIdx.x & 3) ^ 2));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_there) : "r"(recv_bar), "r"((blockIdx.x & 3) ^ 2));
        for (int c = grp * PAIR_CHUNK; c < BN / 2 && t0 + o_beg + c < M && ok; c += PAIR_GROUPS * PAIR_CHUNK) {
          float v[PAIR_CHUNK];
          tmem_ld16(tbase + o_beg + c, v);
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; j += 4)
            asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                         ::"r"(there + (uint32_t)((c + j) / 4 * TC_BM * 16)), "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3]), "r"(bar_there)
                         : "memory");
        }
        if (ok) ok = mbar_wait_cluster(recv_bar, 0);
        if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
        ok = __all_sync(0xffffffffu, ok);
      }
      for (int c = r_beg + grp * PAIR_CHUNK; c < r_end && !direct; c += PAIR_GROUPS * PAIR_CHUNK) {
        if (t0 + c >= M) break;
        float v[PAIR_CHUNK];
#pragma unroll
        for (int j = 0; j < PAIR_CHUNK; j += 16) tmem_ld16(tbase + c + j, v + j);
        if (split == 2) {
          const float4 *from = reinterpret_cast<const float4 *>(smem_raw + (recv0 - smem_u32(smem_raw))) + (c - r_beg) / 4 * TC_BM + fl;
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; j += 4) {
            const float4 p = from[j / 4 * TC_BM];
            v[j] += p.x; v[j + 1] += p.y; v[j + 2] += p.z; v[j + 3] += p.w;
          }
        }
        if (nm.ssq_in) {
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; j += 4) {
            const float4 k = *reinterpret_cast<const float4 *>(scale + c + j);
            v[j] *= k.x; v[j + 1] *= k.y; v[j + 2] *= k.z; v[j + 3] *= k.w;
          }
        }
        if (produce) {
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; ++j) v[j] += old[j];
          fetch_old(c + PAIR_GROUPS * PAIR_CHUNK);
        }
        // the staging tile is free once its previous copy (or the previous chunk's readers) are done
        if (leader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        if (tma_c == SK_TMA_BF16) {
          if (epi == EPI_GELU_T) {
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; j += 2) {
              const uint32_t p = gelu_erf_fast2(v[j], v[j + 1]);
              stage_u[j * TC_BM + fl] = (uint16_t)p;
              stage_u[(j + 1) * TC_BM + fl] = (uint16_t)(p >> 16);
            }
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
        if (pr.rope) {
          if (ok && f0 < N) {
            pair_rope_rows(stage_f, pos + c, cs, w4, pl, f0, t0 + c, M, N, C, pr);
            const int cn = c + PAIR_GROUPS * PAIR_CHUNK;
            if (rotate && cn < BN) pair_rope_fetch(cs, pos + cn, w4, t0 + cn, M, pr.dh >> 1, pl.dim, pr.rope);
          }
          continue;
        }
        if (leader && ok && f0 < N) {
          if (tma_c == SK_TMA_ADD && !produce)
            asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(&mapC), "r"(f0), "r"(t0 + c), "r"(stage) : "memory");
          else
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(&mapC), "r"(f0), "r"(t0 + c), "r"(stage) : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        if (produce && ok && f0 < N) {
          // this warp's four rows: the next contraction's operand and the sums of squares over these 128 features
#pragma unroll
          for (int r = 0; r < PAIR_CHUNK / 4; ++r) {
            const int tl = w4 * (PAIR_CHUNK / 4) + r, t = t0 + c + tl;
            const float4 x = *reinterpret_cast<const float4 *>(stage_f + tl * TC_BM + lane * 4);
            const float sq = warp_sum(fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, x.w * x.w))));
            if (t < M) {
              *reinterpret_cast<uint2 *>(nm.a_out + (size_t)t * N + fc) =
                  make_uint2(pack_bf16x2(gain.x * x.x, gain.y * x.y), pack_bf16x2(gain.z * x.z, gain.w * x.w));
              if (lane == 0) nm.ssq_out[(size_t)t * (N >> 7) + (f0 >> 7)] = sq;
            }
          }
        }
      }
      // accumulator drained: rank 0 may overwrite it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_rank(acc_empty0 + 8 * buf, 2 * half);
        if (nm.ssq_in || pr.rope) mbar_arrive(rows_empty0 + 8 * (i & 1));
      }
    }
    if (leader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();          // no rank leaves while the other's MMAs read its shared memory or its arrivals are under way
  if (warp == PAIR_EPI_WARPS + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------ host side
struct PairShape {
  int BN, stages, n_acc, tmem_cols, pairs, smem_bytes, split;
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

// Tile rule, in cycles: the block steps of the pair with the most tiles (see the header; tiles below 96 tokens gain
// nothing, a step's fixed part shows), the epilogue of a pair's last tile, which nothing hides, and 20 for each pair at
// work: the kernel behind starts on the SMs that are left.  (Chains of one contraction alone, 168 shapes of d = 128 to
// 1280 at 576 to 16320 tokens: 2.0 % above the best tile on average and 15 % at worst, with 10 for a pair 0.6 and 10 %.
// In whole passes 10 is the worse: it gives Wo and W2 64-token tiles on 65 to 68 pairs instead of 96-token ones on 45;
// scoring 800 tokens with d = 1280 333 -> 349 us, 1040 with d = 1024 300 -> 310, decoding 1024 series 2670 -> 2738.)
// can_split (residual updates): where the tiles keep at most half of the pairs busy and K is long, two pairs share a tile, each
// with half of K (32 tiles at most: 128 SMs in clusters of four); the exchange counts 2000 cycles.  Inside forecasts, us: 576 x
// 1280 x 5120 (30 tiles) 18.5 -> 13.4, 1024 x 768 x 3072 (33 -> 24 tiles) 12.9 -> 10.6.  Not where more pairs are busy already
// (1280 x 1024 x 4096, 56: 16.2 -> 15.4 and the next contraction starts later; 1280 x 768 x 3072, 66: 13.6 -> 15.4) and not
// with a short K (576 x 1280 x 1280 10.0 -> 8.5, but the W1 behind it 12.9 -> 13.9; 1280 x 1024 x 1024 9.0 -> 10.1).
static PairShape gemm_pair_geometry(int N, int K, int M, bool can_split = false) {
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
      sh.pairs = tiles;
    }
  }
  sh.split = 1;
  if (can_split && KB >= 32 && sh.pairs <= PAIR_MAX / 2)
    for (int bn = 32; bn <= 256; bn += 32) {
      const int tiles = FT * ((M + bn - 1) / bn);
      const long cost = (KB + 1) / 2 * (256 + (bn < 96 ? 96 : bn)) + 4 * bn + 40 * tiles + 2000;
      if (tiles <= 32 && cost < best) {
        best = cost;
        sh.BN = bn;
        sh.split = 2;
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
  const int recv = sh->split == 2 ? sh->BN / 2 * TC_BM * 4 : 0;
  const int st = (227 * 1024 - PAIR_GROUPS * PAIR_STAGE_OUT - PAIR_ROW_BYTES - 1280 - recv) / stage;
  if (sh->stages == 0) sh->stages = st > PAIR_MAX_STAGES ? PAIR_MAX_STAGES : st;
  sh->smem_bytes = sh->stages * stage + PAIR_GROUPS * PAIR_STAGE_OUT + 1024 + 256 + PAIR_ROW_BYTES + recv;
}

static bool gemm_pair_launch(cudaStream_t st, bool pdl, GemmSkPlan &p, void *C, int M, int epi, int *status, LiveRows lr,
                             const SkNorm *norm = nullptr, const PairRope *rope = nullptr, PairShape sh = PairShape{}) {
  if (M < 1 || M > p.M_max) return false;
  if (!sh.BN) {
    sh = gemm_pair_geometry(p.N, p.K, M, epi == EPI_RESID);
    gemm_pair_fill(&sh, p.N, p.K, M);
  }
  const int idx = sh.BN / 32 - 1;
  if (!p.haveA2[idx]) {
    if (tc_encode(&p.mapA2[idx], p.A, p.M_max, p.K, sh.BN / 2)) return false;
    p.haveA2[idx] = true;
  }
  const int tma_c = epi == EPI_RESID ? SK_TMA_ADD : epi != EPI_F32 ? SK_TMA_BF16 : sh.n_acc == 1 && !rope ? SK_TMA_NONE : SK_TMA_F32;
  const CUtensorMap *mapC = tma_c == SK_TMA_NONE ? &p.mapW : sk_map_c(p, C, M, PAIR_CHUNK, tma_c == SK_TMA_BF16);
  if (!mapC) return false;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * sh.split * sh.pairs);
  cfg.blockDim = dim3(PAIR_THREADS);
  cfg.dynamicSmemBytes = sh.smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2 * sh.split; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel, p.mapW, p.mapA2[idx], *mapC, M, p.N, p.K, sh.BN, sh.split, sh.stages, sh.n_acc,
                            sh.tmem_cols, epi, tma_c, (float *)C, norm ? *norm : SkNorm{}, rope ? *rope : PairRope{}, status,
                            lr) == cudaSuccess;
}

}  // namespace tsfm
