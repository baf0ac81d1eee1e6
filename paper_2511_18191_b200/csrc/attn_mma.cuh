// Causal attention of passes of many tokens on the tensor cores (tcgen05), head size 64, over a bf16 KV cache (which passes:
// attn_mma_pays).
//
// A CTA takes 128 consecutive queries of one (series, head) and walks over the keys they may see in tiles of 128:
//   S = Q K^T (Q in two bf16 parts, high and low, so that the scores keep fp32-like accuracy: eight MMAs of 128 x 128 x 16
//   from shared memory into tensor memory), softmax by two threads per query row, each half of the tile's keys (no shuffle:
//   the row sits in the threads' lane of tensor memory; the two maxima meet in shared memory), probabilities back into tensor
//   memory as bf16, O = P V (P from tensor memory, V as it lies in the cache: the "MN-major" form of the operand), summed over
//   the tiles in registers with the running maximum's factors, as attn_tiles_kernel does it for 16 queries per warp.
// While one CTA's rows are in softmax the other CTA of the SM keeps the tensor core busy (98 KB of shared memory and half of
// tensor memory each).
// Values that a query must not see never meet it: rows behind the last key are zeroed in shared memory, and in tiles that some
// queries see in part, value rows with an infinity or NaN are zeroed too and the queries that do see them set to NaN (a
// product 0 x NaN would reach all 128 queries).  An infinity so makes the head NaN, where in a tile that every query sees it
// stays in its dimension: the token's output is NaN in either case, since the contraction behind multiplies the infinity by
// weights of both signs and the norm behind that by 0.
// Bound: the chain of a tile (MMAs, two passes over the scores, MMAs, sums; 4000 cycles) and a block's start (5000 cycles), with 16
// softmax warps per SM.  A start is one round trip: the queries' loads all leave before the first of them is used and run beside
// the allocation of tensor memory (taken four rows at a time, between stores to shared memory, they were 4500 of 13000 to 16000 cycles
// of a block); outputs leave as rows of 64 bytes by way of shared memory (16 bytes a lane and row before: 1600 cycles).
// us a launch with queries and outputs as before -> now: 64 series x 20 heads x 255 queries 106 -> 84, 64 x 16 x 256 87 -> 68, 16 x 8 x
// 704 36 -> 33.  attn_tiles_kernel -> here: 1280 pairs x 255 queries 112 -> 75, 256 x 256 20 -> 16, 128 x 704 48 -> 34; where which is
// taken: attn_mma_pays.  With one thread per row 14 % slower.
// Warps 0-7 softmax (query row = 32 (w % 4) + lane, keys and output dims of half w / 4), 8 TMA producer, 9 tensor memory and
// MMA issue.  Waits are bounded as in gemm_tc.cuh.  grid = (heads, B, ceil(q_len / 128)), block = 320.
#pragma once
#include "gemm_pair.cuh"
#include "attn_flash.cuh"

namespace tsfm {

constexpr int AM_Q = 128, AM_KEYS = 128, AM_DH = 64;
constexpr int AM_TILE = AM_KEYS * AM_DH * 2;                    // 16 KB: a tile of keys, of values, or one part of the queries
constexpr int AM_WARPS = 8, AM_THREADS = 32 * (AM_WARPS + 2);
constexpr int AM_SMEM = 6 * AM_TILE + 1024 + 128 + 2 * AM_Q * 4;   // Q high, Q low, two stages of K and V
// Shared memory of a launch: two CTAs fit on an SM, but a grid of at most one per SM takes more than half of it, so that no two
// share one while another SM is idle.  (The QKV contraction before it leaves SMs free early, and CTAs that start there pile
// up: see tiles_smem.  Inside forecasts, us a launch with two -> one: 64 pairs x 128 queries behind 770 to 1150 keys 23.7 ->
// 17.5, x 256 behind 1024 to 1792 33.6 -> 25.1, x 256 behind none 10.6 -> 8.0; 128 pairs x 96 behind 770 to 1060 23.7 -> 19.1.)
constexpr int AM_SMEM_ALONE = 114 * 1024;
inline int attn_mma_smem(long ctas) { return ctas <= 148 ? AM_SMEM_ALONE : AM_SMEM; }
constexpr int AM_COLS = 256, AM_S = 0, AM_P = 128, AM_O = 192;   // columns of tensor memory

__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,"
      "%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}

// mapK, mapV: the whole cache as rows of 64 values (box 128 rows); layer_row0: first row of this layer.
__global__ void __launch_bounds__(AM_THREADS, 2)
attn_mma_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, const float *qkv,
                const float2 *__restrict__ rope, PassGeom g, int n_heads, int layer_row0, int rotated, bf16 *out, int *__restrict__ status) {
  extern __shared__ uint8_t am_smem[];
  const uint32_t base = (smem_u32(am_smem) + 1023u) & ~1023u;
  uint8_t *const gbase = am_smem + (base - smem_u32(am_smem));
  const uint32_t q_hi = base, q_lo = base + AM_TILE, ring = base + 2 * AM_TILE, bars = base + 6 * AM_TILE;
  const uint32_t kfull0 = bars, vfull0 = bars + 16, empty0 = bars + 32, q_ready = bars + 48, s_full = bars + 56, p_ready = bars + 64,
                 o_full = bars + 72, slot_addr = bars + 80;
  uint32_t *slot_ptr = reinterpret_cast<uint32_t *>(gbase + 6 * AM_TILE + 80);
  float *half_val = reinterpret_cast<float *>(gbase + 6 * AM_TILE + 128);     // [2][128] what the two threads of a row exchange
  uint32_t *bad_rows = reinterpret_cast<uint32_t *>(gbase + 6 * AM_TILE + 96);   // [4] value rows of the tile with an infinity or NaN
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int h = blockIdx.x, qb = (gridDim.z - 1 - blockIdx.z) * AM_Q, d = n_heads * AM_DH;     // blocks with the most keys first
  const SlotPos sp = slot_lookup(g, blockIdx.y);               // before the dependency wait: see SlotPos
  if (sp.dead) {
    pdl_sync();
    return;
  }
  const int p0 = sp.p0, nq = min(AM_Q, g.q_len - qb);
  const int n_keys = p0 + qb + nq;                             // keys the block's last query sees
  const int n_tiles = (n_keys + AM_KEYS - 1) / AM_KEYS;
  const int row0 = layer_row0 + (sp.b * n_heads + h) * g.cap;

  // TMA producer: tiles of keys that earlier passes left in the cache are requested before the dependency wait
  const bool leader = elect_one();
  auto load = [&](int t) {
    const uint32_t s = (uint32_t)(t & 1), dst = ring + s * 2 * AM_TILE;
    mbar_expect_tx(kfull0 + 8 * s, AM_TILE);
    tma_load_2d(dst, &mapK, 0, row0 + t * AM_KEYS, kfull0 + 8 * s);
    mbar_expect_tx(vfull0 + 8 * s, AM_TILE);
    tma_load_2d(dst + AM_TILE, &mapV, 0, row0 + t * AM_KEYS, vfull0 + 8 * s);
  };
  const int early = min(min(p0 / AM_KEYS, 2), n_tiles);
  // a softmax warp's queries: dims qc .. qc + 3 and their partners 32 further of four rows
  const int qc = (lane & 7) * 4;
  float4 qa[4], qp[4];
  if (warp == AM_WARPS) {
    if (lane < 2) {
      mbar_init(kfull0 + 8 * lane, 1);
      mbar_init(vfull0 + 8 * lane, 1);
      mbar_init(empty0 + 8 * lane, 1);
    }
    if (lane == 0) {
      mbar_init(q_ready, AM_WARPS);
      mbar_init(s_full, 1);
      mbar_init(p_ready, AM_WARPS);
      mbar_init(o_full, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if (leader)
      for (int t = 0; t < early; ++t) load(t);
  } else if (warp == AM_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_addr), "r"((uint32_t)AM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else {
    pdl_sync();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = warp * 16 + i * 4 + (lane >> 3);
      qa[i] = qp[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < nq) {
        const float *src = qkv + ((size_t)blockIdx.y * g.q_len + qb + r) * 3 * d + h * AM_DH + qc;
        qa[i] = __ldcg(reinterpret_cast<const float4 *>(src));
        qp[i] = __ldcg(reinterpret_cast<const float4 *>(src + 32));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot_ptr;

  if (warp == AM_WARPS) {
    // ---------------- TMA producer
    pdl_sync();
    bool ok = true;
    for (int t = early; t < n_tiles && ok; ++t) {
      if (t >= 2) {
        ok = mbar_wait(empty0 + 8 * (t & 1), (uint32_t)(((t >> 1) & 1) ^ 1));
        if (!ok) atomicExch(status, DEV_TIMEOUT_TMA);
      }
      if (leader && ok) load(t);
    }
    __syncwarp();
  } else if (warp == AM_WARPS + 1) {
    // ---------------- MMA issuer (the warp as a whole, one lane issues)
    constexpr uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((AM_KEYS >> 3) << 17) | ((AM_Q >> 4) << 24);
    constexpr uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((AM_DH >> 3) << 17) | ((AM_Q >> 4) << 24);
    pdl_sync();
    const uint64_t dhi = umma_smem_desc(q_hi), dlo = umma_smem_desc(q_lo), dk0 = umma_smem_desc(ring);
    bool ok = mbar_wait(q_ready, 0);
    if (!ok) atomicExch(status, DEV_TIMEOUT_MMA);
    for (int t = 0; t < n_tiles && ok; ++t) {
      const uint32_t s = (uint32_t)(t & 1), ph = (uint32_t)((t >> 1) & 1);
      const uint64_t dk = dk0 + (uint64_t)(s * (2 * AM_TILE >> 4)), dv = dk + (AM_TILE >> 4);
      ok = mbar_wait(kfull0 + 8 * s, ph);
      if (!ok) { atomicExch(status, DEV_TIMEOUT_MMA); break; }
      if (leader) {
#pragma unroll
        for (int k = 0; k < AM_DH / 16; ++k) umma_bf16(tmem + AM_S, dhi + 2 * k, dk + 2 * k, idesc_s, k ? 1u : 0u);
#pragma unroll
        for (int k = 0; k < AM_DH / 16; ++k) umma_bf16(tmem + AM_S, dlo + 2 * k, dk + 2 * k, idesc_s, 1u);
        umma_commit(s_full);
      }
      ok = mbar_wait(p_ready, (uint32_t)(t & 1)) && mbar_wait(vfull0 + 8 * s, ph);
      if (!ok) { atomicExch(status, DEV_TIMEOUT_MMA); break; }
      tc_fence_after();
      if (leader) {
#pragma unroll
        for (int k = 0; k < AM_KEYS / 16; ++k)                 // 16 keys = two groups of eight rows = 2 KB
          umma_bf16_ts(tmem + AM_O, tmem + AM_P + 8 * k, dv + 128 * k, idesc_o, k ? 1u : 0u);
        umma_commit(empty0 + 8 * s);
        umma_commit(o_full);
      }
    }
    __syncwarp();
  } else {
    // ---------------- softmax; first the block's queries: rotated and scaled, high and low parts to shared memory
    {
      const float sc = rsqrtf((float)AM_DH) * 1.4426950408889634f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = warp * 16 + i * 4 + (lane >> 3);
        float4 a = qa[i], b = qp[i];
        if (!rotated && r < nq) {
          const float4 *rp = reinterpret_cast<const float4 *>(rope + (size_t)(p0 + qb + r) * (AM_DH / 2) + qc);
          const float4 cs = rp[0], ct = rp[1];                 // cos sin of dims qc, qc + 1 and qc + 2, qc + 3
          const float4 x = a, y = b;
          a = make_float4((x.x * cs.x - y.x * cs.y) * sc, (x.y * cs.z - y.y * cs.w) * sc, (x.z * ct.x - y.z * ct.y) * sc, (x.w * ct.z - y.w * ct.w) * sc);
          b = make_float4((y.x * cs.x + x.x * cs.y) * sc, (y.y * cs.z + x.y * cs.w) * sc, (y.z * ct.x + x.z * ct.y) * sc, (y.w * ct.z + x.w * ct.w) * sc);
        }
        uint2 hi, lo;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const float4 v = half ? b : a;
          split_bf16x2(v.x, v.y, hi.x, lo.x);
          split_bf16x2(v.z, v.w, hi.y, lo.y);
          const int cc = qc + half * 32;                        // 16-byte chunk cc / 8 of row r sits at chunk ^ (r & 7)
          const uint32_t off = (uint32_t)(r * 128 + (((cc >> 3) ^ (r & 7)) << 4) + (cc & 7) * 2);
          *reinterpret_cast<uint2 *>(gbase + off) = hi;
          *reinterpret_cast<uint2 *>(gbase + AM_TILE + off) = lo;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(q_ready);
    }
    const int w4 = warp & 3, part = warp >> 2;
    const uint32_t trow = tmem + ((uint32_t)(w4 * 32) << 16);
    const int row = w4 * 32 + lane, qpos = p0 + qb + row;      // this thread's query and its position
    float *mine = half_val + part * AM_Q + row, *other = half_val + (part ^ 1) * AM_Q + row;
    uint64_t o[16];                                            // two dims each
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i] = 0;
    float m_run = -INFINITY, l_run = 0.f;
    bool ok = true, nan_seen = false;
    for (int t = 0; t < n_tiles; ++t) {
      const int t0 = t * AM_KEYS, c0 = part * 64, lim = qpos - t0 - c0;      // keys 0 .. lim of this half of the tile are visible
      const bool partial = t0 + AM_KEYS > p0 + qb + 1;         // not all of them to every query (the same for the whole block)
      if (partial) {
        // value rows that some queries must not see: see above
        if (ok) ok = mbar_wait(vfull0 + 8 * (t & 1), (uint32_t)((t >> 1) & 1));
        if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
        if (threadIdx.x < 4) bad_rows[threadIdx.x] = 0;        // none
        asm volatile("bar.sync 1, 256;" ::: "memory");
        uint4 *v = reinterpret_cast<uint4 *>(gbase + 2 * AM_TILE + (t & 1) * 2 * AM_TILE + AM_TILE + row * 128);
        const bool behind = t0 + row >= n_keys;
        if (!behind) {                                         // each thread of a row looks at half of it
          uint32_t bad = 0;                                    // (an exponent of all ones carries into its sign)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 w = v[(i + part * 4 + row) & 7];
            bad |= ((w.x & 0x7f807f80u) + 0x00800080u) | ((w.y & 0x7f807f80u) + 0x00800080u) | ((w.z & 0x7f807f80u) + 0x00800080u) |
                   ((w.w & 0x7f807f80u) + 0x00800080u);
          }
          if (bad & 0x80008000u) atomicOr(bad_rows + (row >> 5), 1u << (row & 31));
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const uint32_t b0 = bad_rows[0], b1 = bad_rows[1], b2 = bad_rows[2], b3 = bad_rows[3];
        const int bad_row = b0 ? __ffs(b0) - 1 : b1 ? 31 + __ffs(b1) : b2 ? 63 + __ffs(b2) : b3 ? 95 + __ffs(b3) : 0x7fffffff;
        if (behind || (bad_rows[row >> 5] >> (row & 31) & 1)) {
#pragma unroll
          for (int i = 0; i < 4; ++i) v[(i + part * 4 + row) & 7] = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        nan_seen |= qpos - t0 >= bad_row;
      }
      if (ok) ok = mbar_wait(s_full, (uint32_t)(t & 1));
      if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
      if (!__all_sync(0xffffffffu, ok)) ok = false;
      tc_fence_after();
      float mx = -INFINITY;
#pragma unroll 1
      for (int c = 0; c < 64; c += 32) {
        float s[32];
        tmem_ld32(trow + AM_S + c0 + c, s);
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (partial) {
#pragma unroll
          for (int i = 0; i < 32; ++i) s[i] = c + i <= lim ? s[i] : -INFINITY;
        }
#pragma unroll
        for (int i = 0; i < 32; i += 2) asm("max.f32 %0, %0, %1, %2;" : "+f"(m4[(i >> 1) & 3]) : "f"(s[i]), "f"(s[i + 1]));
        mx = fmaxf(mx, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
      }
      *mine = mx;
      asm volatile("bar.sync %0, 64;" ::"r"(2 + w4) : "memory");
      const float m_new = fmaxf(m_run, fmaxf(mx, *other)), m_use = m_new == -INFINITY ? 0.f : m_new;
      const float alpha = flash_ex2(m_run - m_use);
      m_run = m_new;
      uint64_t sum2[2] = {0, 0};
      const uint64_t minus_m = f32x2(-m_use, -m_use), alpha2 = f32x2(alpha, alpha);
#pragma unroll 1
      for (int c = 0; c < 64; c += 32) {
        float s[32];
        tmem_ld32(trow + AM_S + c0 + c, s);
        uint32_t p[16];
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float2 x = unpack2(add2(f32x2(s[i], s[i + 1]), minus_m));
          float a = flash_ex2(x.x), b = flash_ex2(x.y);
          if (partial) {
            a = c + i <= lim ? a : 0.f;
            b = c + i + 1 <= lim ? b : 0.f;
          }
          sum2[(i >> 1) & 1] = add2(sum2[(i >> 1) & 1], f32x2(a, b));
          p[i >> 1] = pack_bf16x2(a, b);
        }
        tmem_st16(trow + AM_P + ((c0 + c) >> 1), p);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      const float2 sum = unpack2(add2(sum2[0], sum2[1]));
      l_run = fmaf(l_run, alpha, sum.x + sum.y);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready);
      if (ok) ok = mbar_wait(o_full, (uint32_t)(t & 1));
      if (!ok) atomicExch(status, DEV_TIMEOUT_EPILOGUE);
      if (!__all_sync(0xffffffffu, ok)) ok = false;
      tc_fence_after();
      float v[32];
      tmem_ld32(trow + AM_O + part * 32, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) o[i] = fma2(o[i], alpha2, f32x2(v[2 * i], v[2 * i + 1]));
    }
    *mine = l_run;                                             // (the row's last maxima were read before its last p_ready)
    asm volatile("bar.sync %0, 64;" ::"r"(2 + w4) : "memory");
    // this warp's 32 rows of 64 bytes through shared memory (the queries' MMAs are done), so that four lanes write a row's
    if (ok) {
      const float inv = nan_seen ? __int_as_float(0x7fffffff) : 1.f / (part ? *other + l_run : l_run + *other);
      uint4 *stage = reinterpret_cast<uint4 *>(gbase + warp * 2048);
#pragma unroll
      for (int i = 0; i < 4; ++i) {                            // piece i of row r at i ^ (r / 2 % 4)
        const float2 a = unpack2(o[4 * i]), b = unpack2(o[4 * i + 1]), c = unpack2(o[4 * i + 2]), e = unpack2(o[4 * i + 3]);
        stage[lane * 4 + (i ^ ((lane >> 1) & 3))] = make_uint4(pack_bf16x2(a.x * inv, a.y * inv), pack_bf16x2(b.x * inv, b.y * inv),
                                                               pack_bf16x2(c.x * inv, c.y * inv), pack_bf16x2(e.x * inv, e.y * inv));
      }
      __syncwarp();
      bf16 *dst = out + ((size_t)blockIdx.y * g.q_len + qb + w4 * 32) * d + h * AM_DH + part * 32 + (lane & 3) * 8;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = i * 8 + (lane >> 2);
        const uint4 v = stage[r * 4 + ((lane & 3) ^ ((r >> 1) & 3))];
        if (w4 * 32 + r < nq) *reinterpret_cast<uint4 *>(dst + (size_t)r * d) = v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == AM_WARPS + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)AM_COLS) : "memory");
  }
}

}  // namespace tsfm
