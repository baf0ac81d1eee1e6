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
//   * 16 epilogue warps; a warp takes the 32 features of its lanes of tensor memory in every fourth chunk of 8 or 16 tokens,
//     stages them in two buffers of its own and sends them as boxes of 32 features through the TMA unit (fp32, bf16, added to x):
//     nothing in it waits for another warp.  bf16 results are read from tensor memory in the layout of an mma.sync accumulator,
//     so that stmatrix transposes pairs of tokens into rows of features (2-byte stores to shared memory before: four times the
//     instructions).  What the epilogue of a 256-token tile costs is what decides here: with two accumulators it has to fit under
//     a main loop of 8192 cycles at K = 1024, which alone runs at the tensor rate (512 cycles a K block).  Cycles a tile, groups of
//     four warps sharing a staging tile behind two barriers a chunk -> here: GELU 9400 -> 5800, residual update 12000 (loads and
//     stores from registers) -> 6300, queries 12000 -> 6000; what is left of the contraction's time over its main loop is the last
//     tile's, and the share of L2 that the outputs take (writes 27 bytes a cycle and SM with all SMs writing, reads 60 to 72);
//   * the MMA warp runs its loop as a whole and one lane issues (see gemm_push_kernel): 0.1 to 0.5 us a contraction;
//   * RMSNorms can be folded in (SkNorm; slices of 128 features): a residual epilogue fetches the old rows
//     while the main loop runs, and emits x, the next operand bf16(gain x) and the rows' sums of squares; a
//     consumer scales its rows.  Used where an RMSNorm launch costs more than that (pair_folds);
//   * the QKV contraction of a pass of several query tiles rotates its queries and keys and puts keys and
//     values into the cache as bf16 (PairRope).  Its weight rows are loaded in an order that puts the two members of a rotation
//     pair into one thread (pair_encode_qkv), and the rotation table of the pass's positions sits in shared memory where it
//     fits (pair_table_rows; fetched through L2 a chunk ahead, the queries' tiles took 9500 cycles).
// Scoring passes, us a contraction inside a pass, with shared staging and barriers -> here: M = 6000, d = 1024: QKV 41 -> 34.4, W1 43
// -> 37.2, Wo 17.9 -> 17.9, W2 39 -> 39; M = 5120, d = 768: QKV (fp32) 23.5 -> 20.0, W1 26.5 -> 23.4, Wo 12.7 -> 12.4; M = 4096, d = 512:
// 16.3 -> 16.1, 18.7 -> 14.7, 7.8 -> 7.0, W2 12.0 -> 11.5; M = 16320, d = 1280: QKV 150 -> 133, the rest within the scatter of the clock.
// Plain fp32 outputs of several tiles a pair, staged in boxes of 8 KB -> of 1 KB here: 16384 x 3840 x 1280 123.0 -> 127.8 us, 10500 x 3072 x 1024
// 55.0 -> 55.8, 6000 x 3072 x 1024 32.5 -> 31.9 (boxes of 2 KB 129 .. 140, 57 .. 60, 32 .. 33); of one tile a pair, staged / straight from
// registers, behind W2: 576 x 3840 x 1280 11.5 / 11.8, 1280 x 3072 x 1024 12.2 / 12.7, 1000 x 2304 x 768 8.7 / 9.0.
// Graph replay of dependent launches before the epilogue was per warp, gemm_sk_kernel -> here: M = 16320, d = 1280: QKV 158 -> 118 us
// (1355 TFLOP/s), W1 with GELU 254 -> 160, W2 175 -> 149, Wo 67 -> 50; M = 6000, d = 1024: 47 -> 34, 74 -> 40,
// 61 -> 44, 21 -> 16.
// Warps 0-15 epilogue, 16 TMA producer, 17 tensor-memory allocation and MMA issue, 18-19 the rows' factors and
// cache positions of the next tile.  (With 8 epilogue warps the folded forms, a chain of latencies per chunk, set
// the pace: QKV of 6000 x 1024 60 us.)  Waits are bounded as in gemm_tc.cuh.
#pragma once
#include "gemm_sk.cuh"

namespace tsfm {

// What the epilogue does: fp32 stored; GELU, bf16 stored; fp32 added to what is there; the same with the next norm's operand
// and statistics; rotation and cache append.
enum : int { PAIR_F32 = 0, PAIR_GELU = 1, PAIR_RESID = 2, PAIR_FOLD = 3, PAIR_QKV = 4 };
constexpr int PAIR_CHUNK = 8;                    // tokens that an epilogue warp takes at a time (PAIR_GELU, PAIR_QKV: two chunks)
constexpr int PAIR_GROUPS = 4, PAIR_EPI_WARPS = 4 * PAIR_GROUPS, PAIR_ROW_WARPS = 2;
constexpr int PAIR_THREADS = 32 * (PAIR_EPI_WARPS + 2 + PAIR_ROW_WARPS);
constexpr int PAIR_MAX_STAGES = 8;
constexpr int PAIR_MAX = 74;                     // pairs of SMs on the device
constexpr int PAIR_ROW_BYTES = 2 * 256 * (4 + 8);        // factors and cache positions of two tiles' rows
constexpr int PAIR_FOLD_BYTES = 2 * 4 * 256 * 4;         // (PAIR_FOLD) four warps' sums of squares of two tiles' rows
// Staging of an epilogue warp: two buffers of 8 rows x 32 fp32 or 16 rows x 32 bf16 (PAIR_FOLD: and 8 rows x 32 bf16), or one of
// 16 rows x 32 fp32 (PAIR_QKV).
__host__ __device__ constexpr int pair_stage(int kind) { return kind == PAIR_FOLD ? 3072 : 2048; }

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
// (weights of a QKV contraction: see pair_encode_qkv)
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap *map, int x, int row, int head, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(x), "r"(row), "r"(0), "r"(head), "r"(bar & 0xFEFFFFFFu) : "memory");
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
// Tensor memory in the layout of an mma.sync accumulator: lane / 4 (+ 8) of 16 lanes x columns 2 (lane % 4), + 1 of two blocks of
// eight; a: lanes 0-15, b: lanes 16-31 of the warp's part.  Register 4 block + 2 (lane + 8) + column.
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float (&a)[8], float (&b)[8]) {
  uint32_t r[16];
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr + (16u << 16)) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    a[i] = __uint_as_float(r[i]);
    b[i] = __uint_as_float(r[8 + i]);
  }
}
// Four 8 x 8 blocks of 16-bit values held that way, each transposed: lane 8 m + i gives the address of row i of block m.
__device__ __forceinline__ void stmatrix_trans(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_add_2d(const CUtensorMap *map, int x, int y, uint32_t src) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
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
  int table_rows;                  // (set by gemm_pair_launch) rows of the table that a CTA copies to shared memory: see pair_table_rows
};

// grid = 2 x split x pairs, cluster = 2 x split (split: pairs per tile; residual updates only).  C leaves through mapC (boxes of 32
// features x 8 tokens, PAIR_GELU 16), PAIR_FOLD's next operand through mapA2; the queries of PAIR_QKV are stored to C.
template <int KIND>
__global__ void __launch_bounds__(PAIR_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapA,
                 const __grid_constant__ CUtensorMap mapC, const __grid_constant__ CUtensorMap mapA2, int M, int N, int K, int BN,
                 int split, int stages, int n_acc, int tmem_cols, float *C, const SkNorm nm, const PairRope pr,
                 int *__restrict__ status, const LiveRows lr) {
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
  const uint32_t bars = out0 + PAIR_EPI_WARPS * pair_stage(KIND);
  const uint32_t full0 = bars, empty0 = bars + 64, acc_full0 = bars + 128, acc_empty0 = bars + 144, slot = bars + 160;
  const uint32_t rows_full0 = bars + 176, rows_empty0 = bars + 192, recv_bar = bars + 208;
  const uint32_t recv0 = bars + 256 + PAIR_ROW_BYTES + (KIND == PAIR_FOLD ? PAIR_FOLD_BYTES : 0);   // (split) the other pair's sums of the rows finished here: [quad][feature] x 4 rows
  float *row_scale = reinterpret_cast<float *>(smem_raw + (bars + 256 - smem_u32(smem_raw)));   // [2 tiles][256]
  int2 *row_pos = reinterpret_cast<int2 *>(row_scale + 512);                                    // [2 tiles][256] (cache row of head 0, position)
  float *row_sq = reinterpret_cast<float *>(row_pos + 512);                                     // (PAIR_FOLD) [2 tiles][4 warps][256]
  uint32_t *slot_ptr = reinterpret_cast<uint32_t *>(smem_raw + (slot - smem_u32(smem_raw)));
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int KB_all = (K + TC_BK - 1) / TC_BK, kb0 = KB_all * (int)half / split, KB = KB_all * ((int)half + 1) / split - kb0;
  // rows of the tile that this pair finishes
  const int r_beg = (int)half * (BN / split), r_end = r_beg + BN / split;

  if (warp == PAIR_EPI_WARPS && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapW) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapA) : "memory");
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
      mbar_expect_tx(recv_bar, rows > 0 ? (uint32_t)((rows + PAIR_CHUNK - 1) / PAIR_CHUNK * PAIR_CHUNK * TC_BM * 4) : 0u);
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
      const int dh_log = KIND == PAIR_QKV ? 31 - __clz(pr.dh) : 5;
      auto load_w = [&](uint32_t dst, const Pos &p, uint32_t bar) {
        if constexpr (KIND == PAIR_QKV) {                      // dh / 32 copies
          for (int g = 0, part = TC_W_BYTES >> (dh_log - 5); g < 1 << (dh_log - 5); ++g, dst += part)
            tma_load_4d_pair(dst, &mapW, p.kb * TC_BK, 16 * g, p.wy >> dh_log, bar);
        } else tma_load_2d_pair(dst, &mapW, (kb0 + p.kb) * TC_BK, p.wy, bar);
      };
      Pos pw, pa;
      at_tile(pw, pair);
      pa = pw;
      uint32_t dst = tiles, bar = full0;
      for (int it = 0; it < pre; ++it, dst += stage_bytes, bar += 8, next(pw)) {
        if (rank == 0) mbar_expect_tx(bar, 2u * (uint32_t)stage_bytes);
        load_w(dst, pw, bar);
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
        load_w(dst, pa, full0 + 8 * s);
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
    if (nm.ssq_in || KIND == PAIR_QKV) {
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
          if (KIND == PAIR_QKV) {
            const SlotPos sp = slot_lookup(pr.g, t / pr.g.q_len);
            const int p = sp.p0 + t % pr.g.q_len;
            row_pos[rb * 256 + r] = make_int2(sp.b * pr.n_heads * pr.g.cap + p, p);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(rows_full0 + 8 * rb);
      }
    }
  } else {
    // ---------------- epilogue: a warp has 32 features (its lanes of tensor memory) of every fourth chunk of tokens and its
    // own staging buffers, so that no chunk waits for another warp
    const int grp = warp >> 2, w4 = warp & 3;
    const uint32_t stage = out0 + (uint32_t)(warp * pair_stage(KIND));
    constexpr int CH = KIND == PAIR_GELU || KIND == PAIR_QKV ? 2 * PAIR_CHUNK : PAIR_CHUNK;
    int n_out = 0;                                             // chunks sent so far: their buffers alternate
    // (PAIR_QKV) rotation table: a copy of the rows of the pass's positions (padded by 32 bytes: the four rows that a warp
    // reads at a time lie two apart), or the table itself
    const float2 *table = pr.rope;
    int table_first = 0, table_pitch = pr.dh >> 1;
    if (KIND == PAIR_QKV && pr.table_rows) {
      float2 *copy = reinterpret_cast<float2 *>(smem_raw + (bars + 256 + PAIR_ROW_BYTES - smem_u32(smem_raw)));
      const int vec = pr.dh >> 2;                              // 16-byte pieces of a row
      table_first = pr.g.base;
      table_pitch += 4;
      for (int k = threadIdx.x; k < pr.table_rows * vec; k += 32 * PAIR_EPI_WARPS) {
        const int row = k / vec, v = k - row * vec;
        reinterpret_cast<float4 *>(copy + row * table_pitch)[v] = reinterpret_cast<const float4 *>(pr.rope + (size_t)(table_first + row) * (pr.dh >> 1))[v];
      }
      table = copy;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * PAIR_EPI_WARPS) : "memory");
    }
    pdl_sync();
    bool ok = true;
    for (int tile = pair, i = 0; tile < n_tiles; tile += n_pairs, ++i) {
      const int buf = n_acc == 2 ? (i & 1) : 0, use = n_acc == 2 ? (i >> 1) : i;
      const int f0 = (tile % FT) * 2 * TC_BM + (int)rank * TC_BM, t0 = (tile / FT) * BN;
      const bool mine = f0 < N;                                // (N is a multiple of 128: all of the CTA's features or none)
      const int m_end = mine ? min(M - t0, r_end) : 0;         // rows of the tile to finish here: up to this one
      const float *scale = row_scale + (i & 1) * 256;
      const int2 *pos = row_pos + (i & 1) * 256;
      const int c_beg = r_beg + grp * CH, fw = f0 + w4 * 32;   // first chunk, first feature of this warp
      // (PAIR_FOLD) old values of this warp's first chunk: while the main loop runs
      float old[PAIR_CHUNK], gain = 0.f;
      const float *Cf = C + (size_t)t0 * N + fw + lane;
      auto fetch_old = [&](int c) {
#pragma unroll
        for (int j = 0; j < PAIR_CHUNK; ++j) old[j] = c + j < m_end ? __ldcg(Cf + (size_t)(c + j) * N) : 0.f;
      };
      if (KIND == PAIR_FOLD) {
        fetch_old(c_beg);
        if (mine) gain = nm.gain[fw + lane];
      }
      // (after a wait that ran out: no more waits, nothing stored)
      if (ok && (nm.ssq_in || KIND == PAIR_QKV)) ok = mbar_wait(rows_full0 + 8 * (i & 1), (uint32_t)(i >> 1) & 1u);
      if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
      // (PAIR_QKV) what this tile holds, this warp's dims of it, and the rotation of its first chunk
      const int r = lane >> 2, q = lane & 3;
      int part = 0, f_head = 0, head = 0;                      // queries, keys or values; first of 16 dims in a head; head
      float2 cs[2][2][2];                                      // block of 8 tokens, token, dim r or r + 8
      auto fetch_cs = [&](int c) {
        const float2 *dims = table + f_head + r;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int t = c + 8 * b + 2 * q;
          const int4 p = *reinterpret_cast<const int4 *>(pos + t);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float2 *src = dims + (size_t)((e ? p.w : p.y) - table_first) * table_pitch;
            const bool in = t + e < m_end;
            cs[b][e][0] = in ? src[0] : make_float2(1.f, 0.f);
            cs[b][e][1] = in ? src[8] : make_float2(1.f, 0.f);
          }
        }
      };
      if (KIND == PAIR_QKV && mine) {
        const int d = N / 3, heads = TC_BM / pr.dh;            // (heads of the tile: see pair_encode_qkv)
        part = f0 / d;
        head = (f0 - part * d) / pr.dh + w4 % heads;
        f_head = w4 / heads * 16;
        if (ok && part < 2) fetch_cs(c_beg);
      }
      if (ok) ok = mbar_wait_cluster(acc_full0 + 8 * buf, (uint32_t)use & 1u);
      if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(w4 * 32) << 16) + (uint32_t)(buf * BN);
      if ((KIND == PAIR_RESID || KIND == PAIR_FOLD) && split == 2) {
        // the sums of the rows that the other pair finishes go to the CTA with the same features there (see gemm_push_kernel)
        const int o_beg = BN / 2 - r_beg;                      // (0 or BN / 2)
        uint32_t there, bar_there;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(recv0 + (uint32_t)(w4 * 32 + lane) * 16), "r"((blockIdx.x & 3) ^ 2));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_there) : "r"(recv_bar), "r"((blockIdx.x & 3) ^ 2));
        for (int c = grp * PAIR_CHUNK; c < BN / 2 && t0 + o_beg + c < M && ok; c += PAIR_GROUPS * PAIR_CHUNK) {
          float v[PAIR_CHUNK];
          tmem_ld8(tbase + o_beg + c, v);
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
      for (int c = c_beg; c < m_end && ok; c += PAIR_GROUPS * CH, ++n_out) {
        if (KIND == PAIR_GELU) {
          const uint32_t out = stage + (uint32_t)(n_out & 1) * 1024u;
          float a[8], b[8];
          tmem_ld_frag(tbase + c, a, b);
          uint32_t p[2][4];                                    // block of 8 tokens; features r, r + 8, r + 16, r + 24
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (nm.ssq_in) {
              const float2 s = *reinterpret_cast<const float2 *>(scale + c + 8 * k + 2 * q);
#pragma unroll
              for (int j = 4 * k; j < 4 * k + 4; j += 2) {
                a[j] *= s.x; a[j + 1] *= s.y;
                b[j] *= s.x; b[j + 1] *= s.y;
              }
            }
            p[k][0] = gelu_erf_fast2(a[4 * k], a[4 * k + 1]);
            p[k][1] = gelu_erf_fast2(a[4 * k + 2], a[4 * k + 3]);
            p[k][2] = gelu_erf_fast2(b[4 * k], b[4 * k + 1]);
            p[k][3] = gelu_erf_fast2(b[4 * k + 2], b[4 * k + 3]);
          }
          // the buffer is free once its copy of two chunks ago has read it
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          __syncwarp();
          // rows of 64 bytes; 16-byte piece j of row i at j ^ (i / 2 % 4) (the map's swizzle)
          const uint32_t to = out + (uint32_t)((lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4));
          stmatrix_trans(to, p[0]);
          stmatrix_trans(to + 512, p[1]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&mapC, fw, t0 + c, out);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        } else if (KIND == PAIR_QKV) {
          float a[8], b[8];                                    // dims r, r + 8 of a head's first half, and their partners
          tmem_ld_frag(tbase + c, a, b);
          if (nm.ssq_in) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const float2 s = *reinterpret_cast<const float2 *>(scale + c + 8 * k + 2 * q);
#pragma unroll
              for (int j = 4 * k; j < 4 * k + 4; j += 2) {
                a[j] *= s.x; a[j + 1] *= s.y;
                b[j] *= s.x; b[j + 1] *= s.y;
              }
            }
          }
          if (part < 2) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float2 k = cs[j >> 2][j & 1][(j >> 1) & 1];
              const float x = a[j];
              a[j] = x * k.x - b[j] * k.y;
              b[j] = b[j] * k.x + x * k.y;
            }
            if (c + PAIR_GROUPS * CH < m_end) fetch_cs(c + PAIR_GROUPS * CH);
          }
          __syncwarp();                                        // the previous chunk has been read
          if (part == 0) {
            // fp32 rows of 128 bytes; 16-byte piece j of row i at j ^ (i % 8)
            const float sc = rsqrtf((float)pr.dh) * 1.4426950408889634f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int row = 8 * (j >> 2) + 2 * q + (j & 1), piece = ((r >> 2) + 2 * ((j >> 1) & 1)) ^ (row & 7);
              const uint32_t to = stage + (uint32_t)(row * 128 + (piece << 4) + (r & 3) * 4);
              asm volatile("st.shared.f32 [%0], %1;" ::"r"(to), "f"(a[j] * sc) : "memory");
              asm volatile("st.shared.f32 [%0], %1;" ::"r"(to ^ 64u), "f"(b[j] * sc) : "memory");
            }
            __syncwarp();
            const int row = lane >> 3, j = lane & 7;           // rows lane / 8 + 0, 4, 8, 12; first half of the head: j < 4
            float *dst = C + (size_t)(t0 + c + row) * N + head * pr.dh + (j >> 2) * (pr.dh >> 1) + f_head + (j & 3) * 4;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int rk = row + 4 * k;
              float4 v;
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                           : "r"(stage + (uint32_t)(rk * 128 + ((j ^ (rk & 7)) << 4))) : "memory");
              if (c + rk < m_end) *reinterpret_cast<float4 *>(dst + (size_t)(4 * k) * N) = v;
            }
          } else {
            uint32_t p[2][4];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              p[k][0] = pack_bf16x2(a[4 * k], a[4 * k + 1]);
              p[k][1] = pack_bf16x2(a[4 * k + 2], a[4 * k + 3]);
              p[k][2] = pack_bf16x2(b[4 * k], b[4 * k + 1]);
              p[k][3] = pack_bf16x2(b[4 * k + 2], b[4 * k + 3]);
            }
            const uint32_t to = stage + (uint32_t)((lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4));
            stmatrix_trans(to, p[0]);
            stmatrix_trans(to + 512, p[1]);
            __syncwarp();
            bf16 *cache = (part == 1 ? pr.Kc : pr.Vc) + (size_t)head * pr.g.cap * pr.dh + (q >> 1) * (pr.dh >> 1) + f_head + (q & 1) * 8;
#pragma unroll
            for (int k = 0; k < 2; ++k) {                      // rows r and r + 8, 16-byte piece q
              const int rk = r + 8 * k;
              uint4 v;
              asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                           : "r"(stage + (uint32_t)(rk * 64 + ((q ^ ((rk >> 1) & 3)) << 4))) : "memory");
              if (c + rk < m_end) *reinterpret_cast<uint4 *>(cache + (size_t)pos[c + rk].x * pr.dh) = v;
            }
          }
        } else {
          const uint32_t out = stage + (uint32_t)(n_out & 1) * 1024u, out_a = stage + 2048u + (uint32_t)(n_out & 1) * 512u;
          float v[PAIR_CHUNK];
          tmem_ld8(tbase + c, v);
          if (KIND != PAIR_F32 && split == 2) {
            const float4 *from = reinterpret_cast<const float4 *>(smem_raw + (recv0 - smem_u32(smem_raw))) + (c - r_beg) / 4 * TC_BM + w4 * 32 + lane;
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; j += 4) {
              const float4 p = from[j / 4 * TC_BM];
              v[j] += p.x; v[j + 1] += p.y; v[j + 2] += p.z; v[j + 3] += p.w;
            }
          }
          if (KIND == PAIR_F32 && nm.ssq_in) {
            const float4 k0 = *reinterpret_cast<const float4 *>(scale + c), k1 = *reinterpret_cast<const float4 *>(scale + c + 4);
            v[0] *= k0.x; v[1] *= k0.y; v[2] *= k0.z; v[3] *= k0.w;
            v[4] *= k1.x; v[5] *= k1.y; v[6] *= k1.z; v[7] *= k1.w;
          }
          if (KIND == PAIR_FOLD) {
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; ++j) v[j] += old[j];
            fetch_old(c + PAIR_GROUPS * PAIR_CHUNK);
          }
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          __syncwarp();
#pragma unroll
          for (int j = 0; j < PAIR_CHUNK; ++j) asm volatile("st.shared.f32 [%0], %1;" ::"r"(out + (uint32_t)(j * 128 + lane * 4)), "f"(v[j]) : "memory");
          if (KIND == PAIR_FOLD) {
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; j += 2) {
              const uint32_t p = pack_bf16x2(gain * v[j], gain * v[j + 1]);
              asm volatile("st.shared.u16 [%0], %1;" ::"r"(out_a + (uint32_t)(j * 64 + lane * 2)), "h"((uint16_t)p) : "memory");
              asm volatile("st.shared.u16 [%0], %1;" ::"r"(out_a + (uint32_t)((j + 1) * 64 + lane * 2)), "h"((uint16_t)(p >> 16)) : "memory");
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (KIND == PAIR_RESID) tma_add_2d(&mapC, fw, t0 + c, out);
            else tma_store_2d(&mapC, fw, t0 + c, out);
            if (KIND == PAIR_FOLD) tma_store_2d(&mapA2, fw, t0 + c, out_a);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
          if (KIND == PAIR_FOLD) {
            // the rows' sums of squares over this warp's features: a lane ends with one row
#pragma unroll
            for (int j = 0; j < PAIR_CHUNK; ++j) v[j] *= v[j];
            const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
            float r4[4], r2[2];
#pragma unroll
            for (int j = 0; j < 4; ++j) r4[j] = __shfl_xor_sync(0xffffffffu, b16 ? v[j] : v[j + 4], 16) + (b16 ? v[j + 4] : v[j]);
#pragma unroll
            for (int j = 0; j < 2; ++j) r2[j] = __shfl_xor_sync(0xffffffffu, b8 ? r4[j] : r4[j + 2], 8) + (b8 ? r4[j + 2] : r4[j]);
            float sq = __shfl_xor_sync(0xffffffffu, b4 ? r2[0] : r2[1], 4) + (b4 ? r2[1] : r2[0]);
            sq += __shfl_xor_sync(0xffffffffu, sq, 2);
            sq += __shfl_xor_sync(0xffffffffu, sq, 1);
            if ((lane & 3) == 0) row_sq[((i & 1) * 4 + w4) * 256 + c + (b16 ? 4 : 0) + (b8 ? 2 : 0) + (b4 ? 1 : 0)] = sq;
          }
        }
      }
      // accumulator drained: rank 0 may overwrite it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_rank(acc_empty0 + 8 * buf, 2 * half);
        if (nm.ssq_in || KIND == PAIR_QKV) mbar_arrive(rows_empty0 + 8 * (i & 1));
      }
      if (KIND == PAIR_FOLD) {
        // this group's rows over the CTA's 128 features (the buffer is written again two tiles on, behind the next barrier)
        asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        const int k = w4 * 32 + lane, row = c_beg + (k >> 3) * PAIR_GROUPS * PAIR_CHUNK + (k & 7);
        if (row < m_end && ok) {
          const float *sq = row_sq + (i & 1) * 1024 + row;
          nm.ssq_out[(size_t)(t0 + row) * (N >> 7) + (f0 >> 7)] = (sq[0] + sq[256]) + (sq[512] + sq[768]);
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
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
  for (auto *kernel : {gemm_pair_kernel<PAIR_F32>, gemm_pair_kernel<PAIR_GELU>, gemm_pair_kernel<PAIR_RESID>, gemm_pair_kernel<PAIR_FOLD>,
                       gemm_pair_kernel<PAIR_QKV>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) return -4;
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
// Shapes and outputs it takes: whole 128-feature tiles.
static bool gemm_pair_eligible(const GemmSkPlan &p, const void *C) { return p.valid && p.N % TC_BM == 0 && !((uintptr_t)C & 15); }

// The weights of a QKV contraction [3 d][K] as tiles of 128 features in which the two members of a rotation pair (c and
// c + dh / 2 of a head) are 16 rows apart, i.e. 16 lanes of one epilogue warp: a copy takes 16 rows of both halves of each
// of the tile's heads, dh / 32 copies make a tile.
static int pair_encode_qkv(CUtensorMap *map, const void *base, int N, int K, int dh) {
  const cuuint64_t row = (cuuint64_t)K * 2;
  cuuint64_t dims[4] = {(cuuint64_t)K, (cuuint64_t)(dh / 2), 2, (cuuint64_t)(N / dh)};
  cuuint64_t strides[3] = {row, row * (dh / 2), row * dh};
  cuuint32_t box[4] = {(cuuint32_t)TC_BK, 16, 2, (cuuint32_t)(TC_BM / dh)};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -4;
}

// Rows of the rotation table that a QKV contraction keeps in shared memory: the positions of a pass that starts at the same one in
// every series (prefill, scoring), where they leave room for four stages of the ring.
constexpr int PAIR_TABLE_BYTES = 40 * 1024;
static int pair_table_rows(const PairRope &r) {
  return !r.g.done && r.g.q_len * (r.dh * 4 + 32) <= PAIR_TABLE_BYTES ? r.g.q_len : 0;
}

// Ring depth and tensor memory of a tile width for M tokens.
static void gemm_pair_fill(PairShape *sh, int N, int K, int M, int kind, int table_bytes) {
  const int FT = (N + 2 * TC_BM - 1) / (2 * TC_BM);
  const int tiles = FT * ((M + sh->BN - 1) / sh->BN);
  sh->pairs = tiles < PAIR_MAX ? tiles : PAIR_MAX;
  sh->n_acc = tiles > PAIR_MAX ? 2 : 1;
  const int cols = sh->BN * sh->n_acc;
  sh->tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
  const int stage = TC_W_BYTES + sh->BN / 2 * TC_BK * 2;
  const int rest = 1024 + 256 + PAIR_EPI_WARPS * pair_stage(kind) + PAIR_ROW_BYTES + (kind == PAIR_FOLD ? PAIR_FOLD_BYTES : 0) + table_bytes + (sh->split == 2 ? sh->BN / 2 * TC_BM * 4 : 0);
  const int st = (227 * 1024 - rest) / stage;
  if (sh->stages == 0) sh->stages = st > PAIR_MAX_STAGES ? PAIR_MAX_STAGES : st;
  sh->smem_bytes = sh->stages * stage + rest;
}

static bool gemm_pair_launch(cudaStream_t st, bool pdl, GemmSkPlan &p, void *C, int M, int epi, int *status, LiveRows lr,
                             const SkNorm *norm = nullptr, const PairRope *rope = nullptr, PairShape sh = PairShape{}) {
  if (M < 1 || M > p.M_max) return false;
  if (epi != EPI_F32 && epi != EPI_GELU_T && epi != EPI_RESID) return false;
  const int kind = rope ? PAIR_QKV : epi == EPI_F32 ? PAIR_F32 : epi == EPI_GELU_T ? PAIR_GELU : norm && norm->a_out ? PAIR_FOLD : PAIR_RESID;
  if (!sh.BN) sh = gemm_pair_geometry(p.N, p.K, M, epi == EPI_RESID);
  PairRope pr{};
  if (rope) pr = *rope, pr.table_rows = pair_table_rows(pr);
  gemm_pair_fill(&sh, p.N, p.K, M, kind, pr.table_rows * (pr.dh * 4 + 32));
  const int idx = sh.BN / 32 - 1;
  if (!p.haveA2[idx]) {
    if (tc_encode(&p.mapA2[idx], p.A, p.M_max, p.K, sh.BN / 2)) return false;
    p.haveA2[idx] = true;
  }
  if (rope && p.qkv_dh != rope->dh) {
    if (p.N % 3 || (p.N / 3) % TC_BM || TC_BM % rope->dh || pair_encode_qkv(&p.mapQkv, p.W, p.N, p.K, rope->dh)) return false;
    p.qkv_dh = rope->dh;
  }
  CUtensorMap mapC = p.mapW, mapA2 = p.mapW;
  if (kind != PAIR_QKV && !sk_map_c(p, C, M, kind == PAIR_GELU, kind == PAIR_GELU, &mapC)) return false;
  if (kind == PAIR_FOLD && !sk_map_c(p, norm->a_out, M, true, false, &mapA2)) return false;
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
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, kind == PAIR_QKV ? p.mapQkv : p.mapW, p.mapA2[idx], mapC, mapA2, M, p.N, p.K, sh.BN, sh.split, sh.stages,
                              sh.n_acc, sh.tmem_cols, (float *)C, norm ? *norm : SkNorm{}, pr, status, lr) == cudaSuccess;
  };
  return kind == PAIR_F32 ? go(gemm_pair_kernel<PAIR_F32>) : kind == PAIR_GELU ? go(gemm_pair_kernel<PAIR_GELU>)
         : kind == PAIR_RESID ? go(gemm_pair_kernel<PAIR_RESID>) : kind == PAIR_FOLD ? go(gemm_pair_kernel<PAIR_FOLD>) : go(gemm_pair_kernel<PAIR_QKV>);
}

}  // namespace tsfm
